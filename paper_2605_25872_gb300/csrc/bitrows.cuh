// bitrows.cuh -- the q (or spin) values of one natural x row as an L-bit
// mask, built from the two colour rows of the packed layout (shared by the
// cluster and measurement kernels).
#pragma once

#include "geometry.cuh"

namespace pthr {

// bit m of v -> bit 2m (m < 16)
__device__ __forceinline__ uint32_t spread_bits(uint32_t v) {
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

// bit 2m of v -> bit m
__device__ __forceinline__ uint32_t compact_bits(uint32_t v) {
    v &= 0x55555555u;
    v = (v | (v >> 1)) & 0x33333333u;
    v = (v | (v >> 2)) & 0x0F0F0F0Fu;
    v = (v | (v >> 4)) & 0x00FF00FFu;
    v = (v | (v >> 8)) & 0x0000FFFFu;
    return v;
}

// L-bit row rotated so that bit x holds bit (x + 1) mod L
template <int L>
__device__ __forceinline__ uint32_t rot_next(uint32_t v) {
    return (v >> 1) | ((v & 1u) << (L - 1));
}

// the W words of one colour row
template <int W>
__device__ __forceinline__ void load_words(const uint32_t *p, uint32_t (&w)[W]) {
    if (W == 2) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        w[0] = v.x;
        w[W - 1] = v.y;
    } else {
#pragma unroll
        for (int j = 0; j < W; ++j) w[j] = p[j];
    }
}
template <int W>
__device__ __forceinline__ void store_words(uint32_t *p, const uint32_t (&w)[W]) {
    if (W == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[W - 1]);
    } else {
#pragma unroll
        for (int j = 0; j < W; ++j) p[j] = w[j];
    }
}

// Sign bits (1 = spin -1) of a natural x row whose colour-0 sites have x parity
// p0: the two colour rows interleave (colour c holds x = 2m + p_c).
// From the packed words of the byte layout: a multiply spreads a word's four
// sign bits to every other bit (bits 25, 27, 29, 31 of the product).
template <int L>
__device__ __forceinline__ uint32_t row_of_words(const uint32_t (&w)[2][Geom<L>::W], int p0) {
    constexpr int Lh = L / 2;
    constexpr uint32_t H = 0x55555555u & ((1u << (2 * Lh - 1)) | ((1u << (2 * Lh - 1)) - 1u));
    uint32_t row[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t acc = 0;
#pragma unroll
        for (int j = 0; j < Geom<L>::W; ++j) acc |= (((w[c][j] & 0x80808080u) * 0x00041041u) >> 25) << (8 * j);
        row[c] = acc & H;
    }
    return (row[0] << p0) | (row[1] << (p0 ^ 1));
}
// From the bit layout, row r.
template <int L>
__device__ __forceinline__ uint32_t row_of_bits(const uint32_t *S, int r, int p0) {
    constexpr int W = Geom<L>::W;
    uint32_t row[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t n = 0;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const int w = (c * Geom<L>::ROWS + r) * W + j;
            n |= ((S[w >> 3] >> (4 * (w & 7))) & 0xFu) << (4 * j);
        }
        row[c] = spread_bits(n & ((1u << (L / 2)) - 1u));
    }
    return (row[0] << p0) | (row[1] << (p0 ^ 1));
}

// Row r = y + L z of the bit mask where lattices A and B differ (q_i = -1):
// bit x set iff the spins at x + L r differ.  A and B in the storage layout
// (BITS: the bit layout, else the byte layout).
template <int L, bool BITS>
__device__ __forceinline__ uint32_t diff_row(const uint32_t *A, const uint32_t *B, int r) {
    using Gm = Geom<L>;
    constexpr int W = Gm::W, ROWS = Gm::ROWS;
    const int p0 = ((r % L) + (r / L)) & 1;     // x parity of colour 0 in this row
    if (BITS) return row_of_bits<L>(A, r, p0) ^ row_of_bits<L>(B, r, p0);
    uint32_t w[2][W], v[W];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        load_words<W>(A + (c * ROWS + r) * W, w[c]);
        load_words<W>(B + (c * ROWS + r) * W, v);
#pragma unroll
        for (int j = 0; j < W; ++j) w[c][j] ^= v[j];
    }
    return row_of_words<L>(w, p0);
}

}  // namespace pthr
