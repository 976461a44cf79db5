// Compressed check messages of the streaming variant (FP32 mode, rows of at most 27 edges).
//
// Every message a check sends in one iteration follows from four things (Section III,
// Observations 1 and 2): the two smallest magnitudes min0 <= min1 of the row's lambdas,
// the first location of min0, and per edge the sign (the row's sign parity XOR the sign
// of that edge's lambda). So a row of d <= 27 edges keeps, per frame,
//   m0 = min0, m1 = min1 (binary32), and
//   w  = the edge holding min0 (bits 0 .. 4) | sign of the message to edge t at bit 31 - t,
// and the message to edge t is +-(t = w mod 32 ? m1 : m0), with the magnitude weighted in the
// learned decoder (max(fma(alpha, m, -beta), 0), alpha and beta of the class of edge t's
// bit). Codes on padded rows of 8 slots keep the upper half of such a word, with the location
// in its low bits: w = location (bits 0 .. 4) | sign of the message to edge t at bit 15 - t.
// Twelve, or ten, bytes per row and frame replace four bytes per message slot (8, 16 or the
// row's edges); the arrays are frame-interleaved like every streaming array, element (row i,
// position p) at i Fp + p.
#pragma once

#include <stdint.h>

#include <type_traits>

#include "ldpc_internal.h"  // kCmsgMaxRow

namespace ldpc_impl {

struct CState {
    float* m0;    // [M][Fp]
    float* m1;    // [M][Fp]
    void* w;      // [M][Fp] uint32_t, or uint16_t (half words)
};

// The three arrays laid out one after the other from `base` (12 M Fp bytes).
__host__ __device__ inline CState cstate_at(void* base, int64_t M, int64_t Fp) {
    float* m0 = static_cast<float*>(base);
    return CState{m0, m0 + M * Fp, m0 + 2 * M * Fp};
}

// The half word as a whole one.
__device__ __forceinline__ uint32_t cmsg_whole(uint16_t h) { return (uint32_t)h << 16 | (h & 31u); }

// Magnitude of the message to edge t (before any weighting).
__device__ __forceinline__ float cmsg_mag(float m0, float m1, uint32_t w, int t) {
    return (w & 31u) == (uint32_t)t ? m1 : m0;
}

// The message to edge t: magnitude m (>= 0) with the sign kept at bit 31 - t of w.
__device__ __forceinline__ float cmsg_signed(float m, uint32_t w, int t) {
    return __uint_as_float(__float_as_uint(m) | ((w << t) & 0x80000000u));
}

// The word of a row of d edges; sg: lambda's signs, edge t at bit d - 1 - t. The message signs
// are the row's parity XOR each edge's own.
__device__ __forceinline__ uint32_t cmsg_word(uint32_t sg, int d, uint32_t loc) {
    const uint32_t p = (__popc(sg) & 1) ? 0xffffffffu : 0u;
    return (d ? (sg ^ p) << (32 - d) : 0u) | loc;
}

// Learned weighting of a magnitude: max(fma(alpha, m, -beta), 0) in binary32.
__device__ __forceinline__ float cmsg_weight(float m, float wa, float wb) {
    const float x = __fmaf_rn(wa, m, -wb);
    return x > 0.0f ? x : 0.0f;
}

// The words of V consecutive frames of a row. H: half words, two to a register, the pick and
// the sign taken where they lie.
template <int V, bool H>
struct alignas(H ? (V > 1 ? V * 2 : 2) : V * 4) CWords {
    static constexpr int kReg = H ? (V + 1) / 2 : V;
    using R = typename std::conditional<H && V == 1, uint16_t, uint32_t>::type;
    R w[kReg];
    __device__ __forceinline__ float mag(float m0, float m1, int v, int t) const {
        if constexpr (!H) return cmsg_mag(m0, m1, w[v], t);
        else if (v & 1) return (w[v / 2] & (31u << 16)) == (uint32_t)t << 16 ? m1 : m0;
        else return cmsg_mag(m0, m1, w[v / 2], t);
    }
    // mag (>= 0) with the sign of the message to edge t of frame v
    __device__ __forceinline__ float signed_mag(float m, int v, int t) const {
        if constexpr (!H) return cmsg_signed(m, w[v], t);
        else return cmsg_signed(m, (v & 1) ? (uint32_t)w[v / 2] : (uint32_t)w[v / 2] << 16, t);
    }
    // from the whole words of the frames
    __device__ __forceinline__ void set(const uint32_t (&x)[V]) {
        if constexpr (!H) {
#pragma unroll
            for (int v = 0; v < V; v++) w[v] = x[v];
        } else if constexpr (V == 1) {
            w[0] = (uint16_t)(x[0] >> 16 | (x[0] & 31u));
        } else {
#pragma unroll
            for (int p = 0; p < V / 2; p++)  // the upper halves, then the locations
                w[p] = __byte_perm(x[2 * p], x[2 * p + 1], 0x7632) | (x[2 * p] & 31u) | (x[2 * p + 1] & 31u) << 16;
        }
    }
};

}  // namespace ldpc_impl
