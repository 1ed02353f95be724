// Generated by gen_median27.py: sort9 (28 comparators), the middle ranks of
// two merged lists of 9 (28 comparators, pruned Batcher networks) and the
// median of those and a third list, on two voxels at once: each 32-bit word
// holds two 16-bit values and every comparator is one packed min and max.
#pragma once

// Packed unsigned 16-bit min and max of both halves (sm_90 and later).
__device__ __forceinline__ uint32_t vmin16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t vmax16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// s[k] receives the k-th smallest of v[0..8].
__device__ __forceinline__ void sort9x2(const uint32_t *v, uint32_t *s) {
    uint32_t w[16];
    w[0] = v[0];
    w[1] = v[1];
    w[2] = v[2];
    w[3] = v[3];
    w[4] = v[4];
    w[5] = v[5];
    w[6] = v[6];
    w[7] = v[7];
    w[8] = v[8];
    { const uint32_t t = vmin16x2(w[0], w[1]); w[1] = vmax16x2(w[0], w[1]); w[0] = t; }
    { const uint32_t t = vmin16x2(w[2], w[3]); w[3] = vmax16x2(w[2], w[3]); w[2] = t; }
    { const uint32_t t = vmin16x2(w[4], w[5]); w[5] = vmax16x2(w[4], w[5]); w[4] = t; }
    { const uint32_t t = vmin16x2(w[6], w[7]); w[7] = vmax16x2(w[6], w[7]); w[6] = t; }
    { const uint32_t t = vmin16x2(w[0], w[2]); w[2] = vmax16x2(w[0], w[2]); w[0] = t; }
    { const uint32_t t = vmin16x2(w[1], w[3]); w[3] = vmax16x2(w[1], w[3]); w[1] = t; }
    { const uint32_t t = vmin16x2(w[4], w[6]); w[6] = vmax16x2(w[4], w[6]); w[4] = t; }
    { const uint32_t t = vmin16x2(w[5], w[7]); w[7] = vmax16x2(w[5], w[7]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[1], w[2]); w[2] = vmax16x2(w[1], w[2]); w[1] = t; }
    { const uint32_t t = vmin16x2(w[5], w[6]); w[6] = vmax16x2(w[5], w[6]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[0], w[4]); w[4] = vmax16x2(w[0], w[4]); w[0] = t; }
    { const uint32_t t = vmin16x2(w[1], w[5]); w[5] = vmax16x2(w[1], w[5]); w[1] = t; }
    { const uint32_t t = vmin16x2(w[2], w[6]); w[6] = vmax16x2(w[2], w[6]); w[2] = t; }
    { const uint32_t t = vmin16x2(w[3], w[7]); w[7] = vmax16x2(w[3], w[7]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[2], w[4]); w[4] = vmax16x2(w[2], w[4]); w[2] = t; }
    { const uint32_t t = vmin16x2(w[3], w[5]); w[5] = vmax16x2(w[3], w[5]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[1], w[2]); w[2] = vmax16x2(w[1], w[2]); w[1] = t; }
    { const uint32_t t = vmin16x2(w[3], w[4]); w[4] = vmax16x2(w[3], w[4]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[5], w[6]); w[6] = vmax16x2(w[5], w[6]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[0], w[8]); w[8] = vmax16x2(w[0], w[8]); w[0] = t; }
    { const uint32_t t = vmin16x2(w[4], w[8]); w[8] = vmax16x2(w[4], w[8]); w[4] = t; }
    { const uint32_t t = vmin16x2(w[2], w[4]); w[4] = vmax16x2(w[2], w[4]); w[2] = t; }
    { const uint32_t t = vmin16x2(w[3], w[5]); w[5] = vmax16x2(w[3], w[5]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[6], w[8]); w[8] = vmax16x2(w[6], w[8]); w[6] = t; }
    { const uint32_t t = vmin16x2(w[1], w[2]); w[2] = vmax16x2(w[1], w[2]); w[1] = t; }
    { const uint32_t t = vmin16x2(w[3], w[4]); w[4] = vmax16x2(w[3], w[4]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[5], w[6]); w[6] = vmax16x2(w[5], w[6]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[7], w[8]); w[8] = vmax16x2(w[7], w[8]); w[7] = t; }
    s[0] = w[0];
    s[1] = w[1];
    s[2] = w[2];
    s[3] = w[3];
    s[4] = w[4];
    s[5] = w[5];
    s[6] = w[6];
    s[7] = w[7];
    s[8] = w[8];
}

// Of a[0..8] and b[0..8], each sorted ascending, m[k] receives the value of
// rank 4 + k (0-based) of the 18, k = 0..9.
__device__ __forceinline__ void merge9x2(const uint32_t *a, const uint32_t *b, uint32_t *m) {
    uint32_t w[32];
    w[0] = a[0];
    w[1] = a[1];
    w[2] = a[2];
    w[3] = a[3];
    w[4] = a[4];
    w[5] = a[5];
    w[6] = a[6];
    w[7] = a[7];
    w[8] = a[8];
    w[16] = b[0];
    w[17] = b[1];
    w[18] = b[2];
    w[19] = b[3];
    w[20] = b[4];
    w[21] = b[5];
    w[22] = b[6];
    w[23] = b[7];
    w[24] = b[8];
    w[16] = vmax16x2(w[0], w[16]);
    w[17] = vmax16x2(w[1], w[17]);
    { const uint32_t t = vmin16x2(w[2], w[18]); w[18] = vmax16x2(w[2], w[18]); w[2] = t; }
    { const uint32_t t = vmin16x2(w[3], w[19]); w[19] = vmax16x2(w[3], w[19]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[4], w[20]); w[20] = vmax16x2(w[4], w[20]); w[4] = t; }
    { const uint32_t t = vmin16x2(w[5], w[21]); w[21] = vmax16x2(w[5], w[21]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[6], w[22]); w[22] = vmax16x2(w[6], w[22]); w[6] = t; }
    w[7] = vmin16x2(w[7], w[23]);
    w[8] = vmin16x2(w[8], w[24]);
    { const uint32_t t = vmin16x2(w[8], w[16]); w[16] = vmax16x2(w[8], w[16]); w[8] = t; }
    { const uint32_t t = vmin16x2(w[4], w[8]); w[8] = vmax16x2(w[4], w[8]); w[4] = t; }
    { const uint32_t t = vmin16x2(w[5], w[17]); w[17] = vmax16x2(w[5], w[17]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[6], w[18]); w[18] = vmax16x2(w[6], w[18]); w[6] = t; }
    { const uint32_t t = vmin16x2(w[7], w[19]); w[19] = vmax16x2(w[7], w[19]); w[7] = t; }
    { const uint32_t t = vmin16x2(w[20], w[16]); w[16] = vmax16x2(w[20], w[16]); w[20] = t; }
    w[4] = vmax16x2(w[2], w[4]);
    { const uint32_t t = vmin16x2(w[3], w[5]); w[5] = vmax16x2(w[3], w[5]); w[3] = t; }
    { const uint32_t t = vmin16x2(w[6], w[8]); w[8] = vmax16x2(w[6], w[8]); w[6] = t; }
    { const uint32_t t = vmin16x2(w[7], w[17]); w[17] = vmax16x2(w[7], w[17]); w[7] = t; }
    { const uint32_t t = vmin16x2(w[18], w[20]); w[20] = vmax16x2(w[18], w[20]); w[18] = t; }
    { const uint32_t t = vmin16x2(w[19], w[21]); w[21] = vmax16x2(w[19], w[21]); w[19] = t; }
    w[22] = vmin16x2(w[22], w[16]);
    w[4] = vmax16x2(w[3], w[4]);
    { const uint32_t t = vmin16x2(w[5], w[6]); w[6] = vmax16x2(w[5], w[6]); w[5] = t; }
    { const uint32_t t = vmin16x2(w[7], w[8]); w[8] = vmax16x2(w[7], w[8]); w[7] = t; }
    { const uint32_t t = vmin16x2(w[17], w[18]); w[18] = vmax16x2(w[17], w[18]); w[17] = t; }
    { const uint32_t t = vmin16x2(w[19], w[20]); w[20] = vmax16x2(w[19], w[20]); w[19] = t; }
    w[21] = vmin16x2(w[21], w[22]);
    m[0] = w[4];
    m[1] = w[5];
    m[2] = w[6];
    m[3] = w[7];
    m[4] = w[8];
    m[5] = w[17];
    m[6] = w[18];
    m[7] = w[19];
    m[8] = w[20];
    m[9] = w[21];
}

// The 14th smallest of the 18 values behind m (merge9x2) and of c[0..8], sorted
// ascending: the smallest over i of the largest of i values of c and 14 - i of
// the others.
__device__ __forceinline__ uint32_t median_merged_x2(const uint32_t *m, const uint32_t *c) {
    uint32_t r = m[9];
#pragma unroll
    for (int i = 1; i <= 9; ++i) r = vmin16x2(r, vmax16x2(c[i - 1], m[9 - i]));
    return r;
}
