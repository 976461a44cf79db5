// Training path of the learned (normalised / offset) Min-Sum decoder: an unrolled forward
// of T flooding iterations that keeps, per iteration, only the compressed state of every
// check (min0, min1, the first location of the minimum, the location of the second
// minimum, the sign parity, and one sign bit per edge), and the hand-written adjoint that
// rebuilds each iteration's messages from that state instead of storing them.
//
// Forward iteration t (1-based), per check i and frame (eq. eta_update with the learned
// magnitude): lambda_e = s_j - eta_e; m_e = min1 at the location of the minimum, else
// min0 (Observation 1); g_e = fma(alpha[t][c], m_e, -beta[t][c]) with c the class of bit j;
// eta_e = S_e * max(g_e, 0) with S_e the extrinsic sign (Observation 2); then per bit
// s_j = r_j + sum of eta in ascending row order (eq. lambda_j).
//
// Adjoint of iteration t, given ds^t (loss gradient w.r.t. s^t) and dlambda^(t+1):
//   deta_e = ds^t_j - dlambda^(t+1)_e               (eta_e feeds s^t_j and lambda^(t+1)_e)
//   dg_e = deta_e * S_e if g_e > 0 else 0           (signs are piecewise constant)
//   dalpha[t][c] += dg_e * m_e,  dbeta[t][c] -= dg_e
//   dm_e = dg_e * alpha[t][c] flows to the edge whose |lambda| is m_e: the minimum's
//   location for every other edge, the second minimum's location for the minimum itself
//   (a subgradient through min / argmin): dlambda^t = sign(lambda) * that sum, else 0;
//   ds^(t-1)_j = sum of dlambda^t over the edges of bit j.
// Layout: frame-interleaved, element (row/edge/bit x, frame f) at x * Fp + f; a warp
// covers 32, 64 or 128 consecutive frames of one check or bit (1, 2 or 4 a lane). No pass
// stores messages or their gradients per edge: both are rebuilt from what a row keeps. The saved state of a check is min0,
// min1 and one word: for codes whose rows have at most 16 edges the word also holds the
// row's sign bits (loc | loc2 << 4 | parity << 8 | sign of lambda_k << (16 + k)), so each
// iteration keeps 12 bytes per check and frame; longer rows keep loc | loc2 << 8 |
// parity << 16 and one sign byte per edge.
#include <algorithm>

#include "../../include/ldpc.h"
#include "ldpc_internal.h"

namespace {

using namespace ldpc_impl;

struct TrainWork {
    int32_t Fp;
    float *r, *s, *eta, *ds;
    uint8_t* sg;     // [T][E][Fp] sign bit of lambda (rows of more than 16 edges only)
    float* mn0;      // [T][M][Fp]
    float* mn1;      // [T][M][Fp]
    uint32_t* info;  // [T][M][Fp]: the check's word (see above)
    // backward: sums of the weight gradients [C][2] of iterations g0 + 1 .. (0-based rows from
    // g0 on), in the place of r and s, which only the forward pass uses
    double* gsum;
    int32_t g0;
};

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Carve the workspace; returns the bytes needed (and fills w when base != nullptr).
size_t carve(int32_t M, int32_t N, int64_t E, int32_t F, int32_t T, bool packed, char* base,
             TrainWork* w) {
    const int32_t Fp = (F + 31) & ~31;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        char* p = base ? base + o : nullptr;
        o += al256(bytes);
        return p;
    };
    char* r = take((size_t)N * Fp * 4);
    char* s = take((size_t)N * Fp * 4);
    char* eta = take((size_t)E * Fp * 4);
    take((size_t)E * Fp * 4);  // the gradient pairs of the rows continue behind eta
    char* ds = take((size_t)N * Fp * 4);
    char* sg = packed ? nullptr : take((size_t)T * E * Fp);
    char* mn0 = take((size_t)T * M * Fp * 4);
    char* mn1 = take((size_t)T * M * Fp * 4);
    char* info = take((size_t)T * M * Fp * 4);
    if (w) {
        w->Fp = Fp;
        w->r = (float*)r;
        w->s = (float*)s;
        w->eta = (float*)eta;
        w->ds = (float*)ds;
        w->sg = (uint8_t*)sg;
        w->mn0 = (float*)mn0;
        w->mn1 = (float*)mn1;
        w->info = (uint32_t*)info;
    }
    return o;
}

// [F][N] -> [N][Fp]; frames past F are zero.
__global__ void k_lw_in(const float* src, int F, int N, float* dst, int Fp) {
    __shared__ float tile[32][33];
    const int j0 = blockIdx.x * 32, f0 = blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += blockDim.y) {
        const int f = f0 + y, j = j0 + threadIdx.x;
        tile[y][threadIdx.x] = (f < F && j < N) ? src[(size_t)f * N + j] : 0.0f;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += blockDim.y) {
        const int j = j0 + y, f = f0 + threadIdx.x;
        if (j < N && f < Fp) dst[(size_t)j * Fp + f] = tile[threadIdx.x][y];
    }
}

struct LwArgs {
    const int32_t *row_ptr, *col_idx, *col_ptr, *col_edge;
    const uint8_t* col_class;
    // padded rows of D slots (rows of at most 16 edges)
    const int32_t* ell_col;
    const uint8_t *ell_deg, *ell_cls;
    // row and position in the row of each CSC edge: one word on the padded row layout (rows of
    // at most 16 edges) and for rows of at most 27, else the two arrays
    const int32_t *ell_cslot, *col_row;
    const uint8_t* col_k;
    int32_t dshift;
    int32_t M, N, C, Fp;
    int32_t vrow;  // entry of row i's gradient pair: 2 i (0), or row_ptr[i] (1)
    int64_t E;
    const float *alpha, *beta;  // [T][C]
};

// V consecutive frames of one row, edge or bit: a lane's share of a frame-interleaved row.
template <typename T, int V>
struct alignas(sizeof(T) * V) LV {
    T x[V];
};
template <int V, typename T>
__device__ __forceinline__ LV<T, V> ldv(const T* p) {
    return *reinterpret_cast<const LV<T, V>*>(p);
}
template <int V, typename T>
__device__ __forceinline__ void stv(T* p, const LV<T, V>& v) {
    *reinterpret_cast<LV<T, V>*>(p) = v;
}
// Fields of a check's word.
template <bool PK>
__device__ __forceinline__ int info_loc(uint32_t info) {
    return info & (PK ? 0xf : 0xff);
}
template <bool PK>
__device__ __forceinline__ int info_loc2(uint32_t info) {
    return (info >> (PK ? 4 : 8)) & (PK ? 0xf : 0xff);
}
template <bool PK>
__device__ __forceinline__ uint32_t info_par(uint32_t info) {
    return (info >> (PK ? 8 : 16)) & 1u;
}

// Row and position in the row of CSC edge q.
template <bool PK>
__device__ __forceinline__ void edge_at(const LwArgs& a, int q, int& i, int& k) {
    if (PK || a.ell_cslot) {
        const int slot = __ldg(a.ell_cslot + q);
        i = slot >> a.dshift;
        k = slot & ((1 << a.dshift) - 1);
    } else {
        i = __ldg(a.col_row + q);
        k = __ldg(a.col_k + q);
    }
}

// Eight columns of a padded row from edge k0 on, and the class of an edge from the row's bytes.
__device__ __forceinline__ void load_cols8(const int32_t* p, int (&c)[8]) {
    const int4 x = __ldg(reinterpret_cast<const int4*>(p)), y = __ldg(reinterpret_cast<const int4*>(p) + 1);
    c[0] = x.x, c[1] = x.y, c[2] = x.z, c[3] = x.w;
    c[4] = y.x, c[5] = y.y, c[6] = y.z, c[7] = y.w;
}
template <int D>
struct RowClasses {
    uint32_t x[D ? D / 4 : 1];
    __device__ __forceinline__ void load(const uint8_t* p) {
#pragma unroll
        for (int q = 0; q < D / 4; q++) x[q] = __ldg(reinterpret_cast<const uint32_t*>(p) + q);
    }
    __device__ __forceinline__ int at(int k) const { return (int)(x[D ? k / 4 : 0] >> (k % 4 * 8) & 255u); }
};

// max(fma(alpha, m, -beta), 0) with the sign bit of `flip`.
__device__ __forceinline__ float lw_message(float m, float alpha, float beta, uint32_t flip) {
    const float g = __fmaf_rn(alpha, m, -beta);
    const float mag = g > 0.0f ? g : 0.0f;
    return __uint_as_float(__float_as_uint(mag) ^ (flip & 0x80000000u));
}

// Forward check pass of iteration t with saving; a warp takes one row of 32 V frames. The
// messages of iteration t - 1 are rebuilt from its saved state (12 bytes a row instead of 4
// an edge, and no message is ever written), so the pass reads each edge's s, gathered, and
// the row's state twice 12 bytes. PK: the row's sign bits go to its word (rows of at most 16
// edges), the padded rows are unrolled (D = 8 or 16; D = 0: longer rows), so that an edge's
// position is a constant in every pick, shift and location, and eight gathers are in flight.
// A launch on N=64800, 256 frames: 112 -> 67 us (with three classes of weights), the adjoint's
// row pass, unrolled likewise, 146 -> 82 us; whole training steps 8.5 -> 6.55 ms, and on N=576,
// 4096 frames, 10 iterations, 0.61 -> 0.52 ms (0.53 with the gradients summed in 64 bits). With the posteriors written
// by the bit pass itself, a training step went from 0.87 to 0.61 ms (N=576, 4096 frames, 10
// iterations) and from 12.7 to 8.5 ms (N=64800, 256 frames, 20 iterations: this pass 167 ->
// 108 us, the bit pass with its output 176 -> 84 us a launch).
template <int V, bool FIRST, int D>
__global__ void __launch_bounds__(128, 4) k_lw_check(LwArgs a, TrainWork w, int t) {
    constexpr bool PK = D > 0;
    const int i = blockIdx.x * 4 + (threadIdx.x >> 5);
    const int f0 = (blockIdx.y * 32 + (threadIdx.x & 31)) * V;
    const int Fp = a.Fp;
    if (i >= a.M || f0 >= Fp) return;
    const bool one = a.C == 1;
    int e0 = 0, d, c8[8];
    RowClasses<D> rc;
    if constexpr (PK) {
        d = __ldg(a.ell_deg + i);
        load_cols8(a.ell_col + (size_t)i * D, c8);
        if (!FIRST && !one) rc.load(a.ell_cls + (size_t)i * D);
    } else {
        e0 = __ldg(a.row_ptr + i);
        d = __ldg(a.row_ptr + i + 1) - e0;
    }
    const float* s = FIRST ? w.r : w.s;
    const size_t ri = ((size_t)(t - 1) * a.M + i) * Fp + f0, rp = ri - (size_t)a.M * Fp;
    uint8_t* sg = PK ? nullptr : w.sg + (size_t)(t - 1) * (size_t)a.E * Fp + (size_t)e0 * Fp + f0;
    const float* al = a.alpha + (size_t)(FIRST ? 0 : t - 2) * a.C;
    const float* be = a.beta + (size_t)(FIRST ? 0 : t - 2) * a.C;
    LV<float, V> om0, om1;
    LV<uint32_t, V> oinfo;
    uint32_t osx[V];  // PK: sign of the old message to edge k at bit k
    float al1 = 1.0f, be1 = 0.0f;
    if (!FIRST) {
        om0 = ldv<V>(w.mn0 + rp);
        om1 = ldv<V>(w.mn1 + rp);
        oinfo = ldv<V>(w.info + rp);
        al1 = __ldg(al);
        be1 = __ldg(be);
        if (PK) {
#pragma unroll
            for (int v = 0; v < V; v++) osx[v] = (oinfo.x[v] >> 16) ^ (info_par<PK>(oinfo.x[v]) ? 0xffffu : 0u);
        }
    }
    LV<float, V> min0, min1;
    int loc[V], loc2[V];
    uint32_t par[V], sgw[V];
#pragma unroll
    for (int v = 0; v < V; v++) {
        min0.x[v] = min1.x[v] = __int_as_float(0x7f800000);
        loc[v] = loc2[v] = 0;
        par[v] = sgw[v] = 0;
    }
    auto edge = [&](const int k, const int col, const LV<float, V>& sv) {
            float ak = al1, bk = be1;
            LV<uint8_t, V> sb;
            if (!FIRST) {
                if (!one) {
                    const int cls = PK ? rc.at(k) : (int)__ldg(a.col_class + col);
                    ak = __ldg(al + cls);
                    bk = __ldg(be + cls);
                }
                if (!PK) sb = ldv<V>(sg - (size_t)a.E * Fp + (size_t)k * Fp);
            }
            LV<uint8_t, V> nb;
#pragma unroll
            for (int v = 0; v < V; v++) {
                float lam = sv.x[v];
                if (!FIRST) {
                    const float m = k == info_loc<PK>(oinfo.x[v]) ? om1.x[v] : om0.x[v];
                    const uint32_t flip =
                        PK ? osx[v] << (31 - k) : (info_par<PK>(oinfo.x[v]) ^ sb.x[v]) << 31;
                    lam = lam - lw_message(m, ak, bk, flip);
                }
                const float m = fabsf(lam);
                if (PK) {  // (sgw << 1) | [lambda < 0]: "+ 0" leaves no -0 and no negative NaN
                    sgw[v] = __funnelshift_l(__float_as_uint(lam + 0.0f), sgw[v], 1);
                } else {
                    const uint32_t neg = lam < 0.0f;
                    par[v] ^= neg;
                    nb.x[v] = (uint8_t)neg;
                }
                const bool lt0 = m < min0.x[v], lt1 = m < min1.x[v];
                loc2[v] = lt0 ? loc[v] : lt1 ? k : loc2[v];
                min1.x[v] = lt0 ? min0.x[v] : lt1 ? m : min1.x[v];
                loc[v] = lt0 ? k : loc[v];
                min0.x[v] = lt0 ? m : min0.x[v];
            }
            if (!PK) stv<V>(sg + (size_t)k * Fp, nb);
    };
    if constexpr (PK) {
#pragma unroll
        for (int k0 = 0; k0 < D; k0 += 8) {
            if (k0 >= d) break;  // the same for the whole warp
            LV<float, V> sv[8];
#pragma unroll
            for (int u = 0; u < 8; u++)
                if (k0 + u < d) sv[u] = ldv<V>(s + (size_t)c8[u] * Fp + f0);
            if (k0 + 8 < D) load_cols8(a.ell_col + (size_t)i * D + k0 + 8, c8);
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (k0 + u >= d) break;
                edge(k0 + u, 0, sv[u]);
            }
        }
    } else {
        constexpr int U = 4;  // gathers in flight together
        for (int k0 = 0; k0 < d; k0 += U) {
            int c[U];
            LV<float, V> sv[U];
#pragma unroll
            for (int u = 0; u < U; u++) c[u] = __ldg(a.col_idx + e0 + min(k0 + u, d - 1));
#pragma unroll
            for (int u = 0; u < U; u++) sv[u] = ldv<V>(s + (size_t)c[u] * Fp + f0);
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (k0 + u >= d) break;
                edge(k0 + u, c[u], sv[u]);
            }
        }
    }
    LV<uint32_t, V> info;
#pragma unroll
    for (int v = 0; v < V; v++) {
        if (PK) sgw[v] = d ? __brev(sgw[v]) >> (32 - d) : 0u;  // the sign of lambda_k to bit k
        info.x[v] = PK ? (uint32_t)loc[v] | ((uint32_t)loc2[v] << 4) | ((__popc(sgw[v]) & 1u) << 8) | (sgw[v] << 16)
                       : (uint32_t)loc[v] | ((uint32_t)loc2[v] << 8) | (par[v] << 16);
    }
    stv<V>(w.mn0 + ri, min0);
    stv<V>(w.mn1 + ri, min1);
    stv<V>(w.info + ri, info);
}

// Tile of 32 bits x 32 V frames between the frame-interleaved arrays (a warp holds one bit,
// a lane V consecutive frames) and the caller's frame-major [F][N] ones: frame lane V + v of
// a bit sits at column v 32 + lane, so neither side has bank conflicts.
template <int V>
struct LwTile {
    float x[32][32 * V + 1];
    __device__ __forceinline__ void put(int c, int lane, const LV<float, V>& a) {
#pragma unroll
        for (int v = 0; v < V; v++) x[c][v * 32 + lane] = a.x[v];
    }
    __device__ __forceinline__ LV<float, V> get(int c, int lane) const {
        LV<float, V> a;
#pragma unroll
        for (int v = 0; v < V; v++) a.x[v] = x[c][v * 32 + lane];
        return a;
    }
    __device__ __forceinline__ float& at(int c, int f) { return x[c][(f % V) * 32 + f / V]; }
};

// Forward bit pass: s = r + sum of eta in ascending row order, the messages rebuilt from the
// rows' states; a block takes 32 bits, 8 warps of 4. soft (nullable): also written to
// soft [F][N], from the tile in shared memory, so that s is not read again to transpose it;
// keep: s is needed by a later iteration.
template <int V, bool PK>
__global__ void __launch_bounds__(256) k_lw_var(LwArgs a, TrainWork w, int t, float* soft, int F, int keep) {
    __shared__ LwTile<V> tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * 32, fb = blockIdx.y * 32 * V, f0 = fb + lane * V;
    const int Fp = a.Fp;
    const size_t base = (size_t)(t - 1) * a.M * Fp + f0;
    for (int b = warp; b < 32 && j0 + b < a.N; b += 8) {
        if (f0 >= Fp) break;
        const int j = j0 + b;
        const int cls = a.C == 1 ? 0 : __ldg(a.col_class + j);
        const float al = __ldg(a.alpha + (size_t)(t - 1) * a.C + cls);
        const float be = __ldg(a.beta + (size_t)(t - 1) * a.C + cls);
        LV<float, V> acc = ldv<V>(w.r + (size_t)j * Fp + f0);
        const int q1 = __ldg(a.col_ptr + j + 1);
#pragma unroll 2
        for (int q = __ldg(a.col_ptr + j); q < q1; q++) {
            int i, k;
            edge_at<PK>(a, q, i, k);
            const size_t o = base + (size_t)i * Fp;
            const LV<float, V> m0 = ldv<V>(w.mn0 + o), m1 = ldv<V>(w.mn1 + o);
            const LV<uint32_t, V> x = ldv<V>(w.info + o);
            LV<uint8_t, V> sb;
            if (!PK)
                sb = ldv<V>(w.sg + ((size_t)(t - 1) * a.E + __ldg(a.col_edge + q)) * Fp + f0);
#pragma unroll
            for (int v = 0; v < V; v++) {
                const float m = k == info_loc<PK>(x.x[v]) ? m1.x[v] : m0.x[v];
                const uint32_t neg = PK ? x.x[v] >> (16 + k) : (uint32_t)sb.x[v];
                acc.x[v] = acc.x[v] + lw_message(m, al, be, (info_par<PK>(x.x[v]) ^ neg) << 31);
            }
        }
        if (keep) stv<V>(w.s + (size_t)j * Fp + f0, acc);
        if (soft) tile.put(b, lane, acc);
    }
    if (!soft) return;
    __syncthreads();
    if (j0 + lane >= a.N) return;
    for (int y = warp; y < 32 * V && fb + y < F; y += 8)
        soft[(size_t)(fb + y) * a.N + j0 + lane] = tile.at(lane, y);
}

// Adjoint of the check pass of iteration t; LAST: t = T (no dlambda^(t+1)). A warp covers
// 32 V frames of one row after another, so the weight gradients collect over many rows
// before they leave the block.
//
// dlambda^t of a row is zero but at the locations of its two minima, so a row keeps two values
// per frame (at loc and at loc2, lambda's sign applied) instead of one per edge; the
// locations are in the saved word. Row i's pair sits at entries 2 i and 2 i + 1 of the
// message region, which the backward pass does not need otherwise (row_ptr[i] and
// row_ptr[i] + 1 when the code has more rows than edges: a row with edges has at least two).
//
// Weight gradients: GM = 0 (one class) in two registers a lane; GM = 1 (at most kLwClasses
// classes) in a shared-memory accumulator of the lane's own per class; GM = 2 by a warp
// reduction and two shared-memory atomics per edge.
//
// One edge and frame a thread with a dense edge gradient and two shared-memory atomics per
// edge was bound by those atomics (all lanes on one address) and by 4-byte loads. Measured,
// whole training steps (forward and backward): N=576, 4096 frames, 10 iterations 3.89 -> 0.87
// ms; N=64800, 256 frames, 20 iterations 38.4 -> 12.7 ms.
constexpr int kLwClasses = 16;
template <int V, bool LAST, int D, int GM>
__global__ void __launch_bounds__(128, 4) k_lw_bwd_row(LwArgs a, TrainWork w, int t) {
    constexpr bool PK = D > 0;
    extern __shared__ float gacc[];  // GM 0, 1: [2 C][128]; GM 2: [2 C]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < 2 * a.C * (GM == 2 ? 1 : 128); q += 128) gacc[q] = 0.0f;
    __syncthreads();
    const int Fp = a.Fp;
    const int f0 = (blockIdx.y * 32 + lane) * V;
    const bool on = f0 < Fp;  // lanes behind the last frame stay for the reductions
    const int fo = on ? f0 : 0;
    const float* al = a.alpha + (size_t)(t - 1) * a.C;
    const float* be = a.beta + (size_t)(t - 1) * a.C;
    const uint8_t* sg = PK ? nullptr : w.sg + (size_t)(t - 1) * (size_t)a.E * Fp;
    float ga = 0.0f, gb = 0.0f;
    for (int i = blockIdx.x * 4 + warp; i < a.M; i += gridDim.x * 4) {
        int e0 = 0, d, c8[8];
        RowClasses<D> rc;
        if constexpr (PK) {
            d = __ldg(a.ell_deg + i);
            load_cols8(a.ell_col + (size_t)i * D, c8);
            if (GM != 0) rc.load(a.ell_cls + (size_t)i * D);
            if (a.vrow) e0 = __ldg(a.row_ptr + i);
        } else {
            e0 = __ldg(a.row_ptr + i);
            d = __ldg(a.row_ptr + i + 1) - e0;
        }
        if (d == 0) continue;
        const size_t ri = ((size_t)(t - 1) * a.M + i) * Fp + fo;
        const size_t rv = (a.vrow ? (size_t)e0 : 2 * (size_t)i) * Fp + fo;
        const LV<float, V> m0 = ldv<V>(w.mn0 + ri), m1 = ldv<V>(w.mn1 + ri);
        const LV<uint32_t, V> info = ldv<V>(w.info + ri);
        LV<float, V> p1, p2;  // dlambda^(t+1) of the row, at that iteration's minima
        LV<uint32_t, V> pinfo;
        if (!LAST) {
            p1 = ldv<V>(w.eta + rv);
            p2 = ldv<V>(w.eta + rv + Fp);
            pinfo = ldv<V>(w.info + ri + (size_t)a.M * Fp);
        }
        float acc1[V], acc2[V];
        uint32_t neg1[V], neg2[V];  // lambda's sign at loc and loc2
        uint32_t sx[V];             // PK: the sign of the message to edge k at bit k
#pragma unroll
        for (int v = 0; v < V; v++) {
            acc1[v] = acc2[v] = 0.0f;
            neg1[v] = neg2[v] = sx[v] = 0;
            if (PK) {
                const uint32_t x = info.x[v];
                sx[v] = (x >> 16) ^ (info_par<PK>(x) ? 0xffffu : 0u);
                neg1[v] = (x >> (16 + info_loc<PK>(x))) & 1u;
                neg2[v] = (x >> (16 + info_loc2<PK>(x))) & 1u;
            }
        }
        auto edge = [&](const int k, const int col, const LV<float, V>& dv) {
                const int cls = GM == 0 ? 0 : PK ? rc.at(k) : (int)__ldg(a.col_class + col);
                const float alpha = __ldg(al + cls), beta = __ldg(be + cls);
                LV<uint8_t, V> sv;
                if (!PK) sv = ldv<V>(sg + (size_t)(e0 + k) * Fp + fo);
                float xa = 0.0f, xb = 0.0f;
#pragma unroll
                for (int v = 0; v < V; v++) {
                    float deta = dv.x[v];
                    if (!LAST)
                        deta -= k == info_loc<PK>(pinfo.x[v])    ? p1.x[v]
                                : k == info_loc2<PK>(pinfo.x[v]) ? p2.x[v]
                                                                 : 0.0f;
                    const bool at0 = k == info_loc<PK>(info.x[v]);
                    const float m = at0 ? m1.x[v] : m0.x[v];
                    const bool pos = __fmaf_rn(alpha, m, -beta) > 0.0f;
                    uint32_t flip;
                    if (PK) {
                        flip = sx[v] << (31 - k);
                    } else {
                        if (at0) neg1[v] = sv.x[v];
                        if (k == info_loc2<PK>(info.x[v])) neg2[v] = sv.x[v];
                        flip = (info_par<PK>(info.x[v]) ^ sv.x[v]) << 31;
                    }
                    const float dg = __uint_as_float(__float_as_uint(deta) ^ (flip & 0x80000000u));
                    const float da = pos ? dg * alpha : 0.0f;
                    acc1[v] += at0 ? 0.0f : da;
                    acc2[v] += at0 ? da : 0.0f;
                    xa += pos ? dg * m : 0.0f;
                    xb -= pos ? dg : 0.0f;
                }
                if constexpr (GM == 0) {
                    ga += xa;
                    gb += xb;
                } else if constexpr (GM == 1) {
                    float* g = gacc + 2 * cls * 128 + threadIdx.x;
                    g[0] += xa;
                    g[128] += xb;
                } else {
                    xa = on ? xa : 0.0f;
                    xb = on ? xb : 0.0f;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        xa += __shfl_xor_sync(0xffffffffu, xa, o);
                        xb += __shfl_xor_sync(0xffffffffu, xb, o);
                    }
                    if (lane == 0) {
                        atomicAdd(gacc + 2 * cls, xa);
                        atomicAdd(gacc + 2 * cls + 1, xb);
                    }
                }
        };
        if constexpr (PK) {
#pragma unroll
            for (int k0 = 0; k0 < D; k0 += 8) {
                if (k0 >= d) break;  // the same for the whole warp
                LV<float, V> dv[8];
#pragma unroll
                for (int u = 0; u < 8; u++)
                    if (k0 + u < d) dv[u] = ldv<V>(w.ds + (size_t)c8[u] * Fp + fo);
                if (k0 + 8 < D) load_cols8(a.ell_col + (size_t)i * D + k0 + 8, c8);
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    if (k0 + u >= d) break;
                    edge(k0 + u, 0, dv[u]);
                }
            }
        } else {
            constexpr int U = 4;  // gathers in flight together
            for (int k0 = 0; k0 < d; k0 += U) {
                int c[U];
                LV<float, V> dv[U];
#pragma unroll
                for (int u = 0; u < U; u++) c[u] = __ldg(a.col_idx + e0 + min(k0 + u, d - 1));
#pragma unroll
                for (int u = 0; u < U; u++) dv[u] = ldv<V>(w.ds + (size_t)c[u] * Fp + fo);
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (k0 + u >= d) break;
                    edge(k0 + u, c[u], dv[u]);
                }
            }
        }
        if (on) {
            LV<float, V> o1, o2;
#pragma unroll
            for (int v = 0; v < V; v++) {  // d|lambda| / dlambda = sign(lambda), sign(0) = +1
                o1.x[v] = neg1[v] ? -acc1[v] : acc1[v];
                o2.x[v] = neg2[v] ? -acc2[v] : acc2[v];
            }
            stv<V>(w.eta + rv, o1);
            stv<V>(w.eta + rv + Fp, o2);
        }
    }
    if constexpr (GM == 0) {
        gacc[threadIdx.x] = ga;
        gacc[128 + threadIdx.x] = gb;
    }
    if (GM != 2 && !on)  // what the lanes behind the last frame added up is not theirs
        for (int q = 0; q < 2 * a.C; q++) gacc[q * 128 + threadIdx.x] = 0.0f;
    __syncthreads();
    for (int q = GM == 2 ? (int)threadIdx.x : warp; q < 2 * a.C; q += GM == 2 ? 128 : 4) {
        // the blocks' sums, some thousand of them, meet in 64 bits
        float x;
        if constexpr (GM == 2) {
            x = gacc[q];
        } else {
            const float* g = gacc + q * 128 + lane;
            x = (g[0] + g[32]) + (g[64] + g[96]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        }
        if (x != 0.0f && (GM == 2 || lane == 0))
            atomicAdd(w.gsum + ((size_t)(t - 1 - w.g0) * a.C + q / 2) * 2 + (q & 1), (double)x);
    }
}

// The summed weight gradients, rounded once.
__global__ void k_lw_grad(const double* __restrict__ gsum, float* grad_alpha, float* grad_beta, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    grad_alpha[i] = (float)gsum[2 * i];
    grad_beta[i] = (float)gsum[2 * i + 1];
}

// ds^(t-1)_j = sum over the edges of bit j of dlambda^t, ascending rows (the pair of each
// row, picked by the row's locations), plus the loss gradient of the posteriors of iteration
// t - 1 (grad [F][N], nullable), read through the tile: a block takes 32 bits. Measured
// against a pass of its own that adds the gradient: 137 + 52 -> 82 us a launch (N=64800, 256
// frames).
template <int V, bool PK>
__global__ void __launch_bounds__(256) k_lw_bwd_col(LwArgs a, TrainWork w, int t, const float* grad, int F) {
    __shared__ LwTile<V> tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * 32, fb = blockIdx.y * 32 * V, f0 = fb + lane * V;
    const int Fp = a.Fp;
    if (grad) {
#pragma unroll 4
        for (int y = warp; y < 32 * V; y += 8)
            tile.at(lane, y) = (fb + y < F && j0 + lane < a.N) ? grad[(size_t)(fb + y) * a.N + j0 + lane] : 0.0f;
        __syncthreads();
    }
    if (f0 >= Fp) return;
    const uint32_t* info = w.info + (size_t)(t - 1) * a.M * Fp;
    for (int b = warp; b < 32 && j0 + b < a.N; b += 8) {
        const int j = j0 + b;
        LV<float, V> acc;
#pragma unroll
        for (int v = 0; v < V; v++) acc.x[v] = 0.0f;
        const int q1 = __ldg(a.col_ptr + j + 1);
#pragma unroll 2
        for (int q = __ldg(a.col_ptr + j); q < q1; q++) {
            int i, k;
            edge_at<PK>(a, q, i, k);
            const size_t rv = (a.vrow ? (size_t)__ldg(a.row_ptr + i) : 2 * (size_t)i) * Fp + f0;
            const LV<uint32_t, V> x = ldv<V>(info + (size_t)i * Fp + f0);
            const LV<float, V> p1 = ldv<V>(w.eta + rv), p2 = ldv<V>(w.eta + rv + Fp);
#pragma unroll
            for (int v = 0; v < V; v++)
                acc.x[v] += k == info_loc<PK>(x.x[v])    ? p1.x[v]
                            : k == info_loc2<PK>(x.x[v]) ? p2.x[v]
                                                         : 0.0f;
        }
        if (grad) {
            const LV<float, V> g = tile.get(b, lane);
#pragma unroll
            for (int v = 0; v < V; v++) acc.x[v] = acc.x[v] + g.x[v];
        }
        stv<V>(w.ds + (size_t)j * Fp + f0, acc);
    }
}

// Frames a lane takes: the widest vector (16 bytes) that still gives the GPU eight warps per SM
// over `rows` rows, and no lane group without frames. One frame when the caller's workspace
// is not 16-byte aligned.
int lane_frames(int32_t rows, int32_t Fp, int num_sms, const void* work) {
    int V = ((uintptr_t)work & 15) ? 1 : 4;
    while (V > 1 && (Fp < 32 * V || (int64_t)rows * ((Fp + 32 * V - 1) / (32 * V)) < 8ll * num_sms)) V /= 2;
    return V;
}

// D: slots of a padded row (0: rows of more than 16 edges).
template <int V, int D>
void launch_fwd(const LwArgs& a, const TrainWork& w, int t, float* soft, int frames, bool keep,
                cudaStream_t st) {
    const int fb = (a.Fp + 32 * V - 1) / (32 * V);
    const dim3 gc((a.M + 3) / 4, fb);
    if (t == 1) k_lw_check<V, true, D><<<gc, 128, 0, st>>>(a, w, t);
    else k_lw_check<V, false, D><<<gc, 128, 0, st>>>(a, w, t);
    k_lw_var<V, (D > 0)><<<dim3((a.N + 31) / 32, fb), 256, 0, st>>>(a, w, t, soft, frames, keep);
}

// grad_prev (nullable): the loss gradient of the posteriors of iteration t - 1.
template <int V, int D>
void launch_bwd(const LwArgs& a, const TrainWork& w, int t, bool last, int num_sms, const float* grad_prev,
                int frames, cudaStream_t st) {
    const int fb = (a.Fp + 32 * V - 1) / (32 * V);
    // about 16 blocks an SM (their warps take several rows each)
    const int gx = std::max(1, std::min((a.M + 3) / 4, (16 * num_sms + fb - 1) / fb));
    const int gm = a.C == 1 ? 0 : a.C <= kLwClasses ? 1 : 2;
    const size_t sm = (size_t)2 * a.C * (gm == 2 ? 1 : 128) * sizeof(float);
    auto go = [&](auto row) { row<<<dim3(gx, fb), 128, sm, st>>>(a, w, t); };
    if (last) {
        if (gm == 0) go(k_lw_bwd_row<V, true, D, 0>);
        else if (gm == 1) go(k_lw_bwd_row<V, true, D, 1>);
        else go(k_lw_bwd_row<V, true, D, 2>);
    } else {
        if (gm == 0) go(k_lw_bwd_row<V, false, D, 0>);
        else if (gm == 1) go(k_lw_bwd_row<V, false, D, 1>);
        else go(k_lw_bwd_row<V, false, D, 2>);
    }
    if (t > 1) k_lw_bwd_col<V, (D > 0)><<<dim3((a.N + 31) / 32, fb), 256, 0, st>>>(a, w, t, grad_prev, frames);
}

// Rows of at most 16 edges (the padded layout) keep their sign bits in the check's word.
bool packed_signs(const HandleView& v) { return v.dg->ell_D > 0; }

int check_common(const HandleView& v, int32_t frames, int32_t iters, const void* alpha,
                 const void* beta, const void* work, uint64_t work_bytes) {
    if (frames <= 0 || iters <= 0 || frames > 65535 * 32) return LDPC_ERR_INVALID_ARG;
    if (!alpha || !beta || !work) return LDPC_ERR_BAD_POINTER;
    if (v.dg->n_classes <= 0 || v.dg->max_dc > 255) return LDPC_ERR_UNSUPPORTED;
    const size_t need = carve(v.M, v.N, v.E, frames, iters, packed_signs(v), nullptr, nullptr);
    if (work_bytes < need) return LDPC_ERR_INVALID_ARG;
    return LDPC_OK;
}

LwArgs make_args(const HandleView& v, int32_t Fp, const float* alpha, const float* beta) {
    LwArgs a;
    a.row_ptr = v.dg->row_ptr;
    a.col_idx = v.dg->col_idx;
    a.col_ptr = v.dg->col_ptr;
    a.col_edge = v.dg->col_edge;
    a.col_class = v.dg->col_class;
    a.ell_col = v.dg->ell_col;
    a.ell_deg = v.dg->ell_deg;
    a.ell_cls = v.dg->ell_cls;
    a.ell_cslot = v.dg->ell_D ? v.dg->ell_cslot : v.dg->row_slot;
    a.col_row = v.dg->col_row;
    a.col_k = v.dg->col_k;
    a.dshift = v.dg->ell_D == 16 ? 4 : v.dg->ell_D == 8 ? 3 : kRowSlotShift;
    a.vrow = v.M > v.E;
    a.M = v.M;
    a.N = v.N;
    a.C = v.dg->n_classes;
    a.Fp = Fp;
    a.E = v.E;
    a.alpha = alpha;
    a.beta = beta;
    return a;
}

}  // namespace

extern "C" {

int ldpc_train_workspace_size(ldpc_t* h, int32_t frames, int32_t iters, uint64_t* bytes) {
    HandleView v;
    if (handle_view(h, &v) != LDPC_OK || !bytes) return LDPC_ERR_BAD_POINTER;
    if (frames <= 0 || iters <= 0) return LDPC_ERR_INVALID_ARG;
    *bytes = carve(v.M, v.N, v.E, frames, iters, packed_signs(v), nullptr, nullptr);
    return LDPC_OK;
}

int ldpc_train_forward(ldpc_t* h, const float* llr, int32_t frames, int32_t iters,
                       const float* alpha, const float* beta, float* soft, int32_t soft_every,
                       void* work, uint64_t work_bytes) {
    HandleView v;
    if (handle_view(h, &v) != LDPC_OK || !llr || !soft) return LDPC_ERR_BAD_POINTER;
    int rc = check_common(v, frames, iters, alpha, beta, work, work_bytes);
    if (rc != LDPC_OK) return rc;
    TrainWork w;
    const bool pk = packed_signs(v);
    carve(v.M, v.N, v.E, frames, iters, pk, (char*)work, &w);
    const LwArgs a = make_args(v, w.Fp, alpha, beta);
    cudaStream_t st = v.stream;
    k_lw_in<<<dim3((v.N + 31) / 32, w.Fp / 32), dim3(32, 8), 0, st>>>(llr, frames, v.N, w.r, w.Fp);
    const int V = lane_frames(v.M, w.Fp, v.num_sms, work);
    const int D = v.dg->ell_D;  // (set exactly where the signs are packed)
    auto step = V == 4   ? (D == 8 ? launch_fwd<4, 8> : D == 16 ? launch_fwd<4, 16> : launch_fwd<4, 0>)
                : V == 2 ? (D == 8 ? launch_fwd<2, 8> : D == 16 ? launch_fwd<2, 16> : launch_fwd<2, 0>)
                         : (D == 8 ? launch_fwd<1, 8> : D == 16 ? launch_fwd<1, 16> : launch_fwd<1, 0>);
    int launches = 1;
    for (int t = 1; t <= iters; t++) {
        float* out = soft_every ? soft + (size_t)(t - 1) * frames * v.N : t == iters ? soft : nullptr;
        step(a, w, t, out, frames, t < iters, st);
        launches += 2;
    }
    *v.last_launches = launches;
    return cudaGetLastError() == cudaSuccess ? LDPC_OK : LDPC_ERR_CUDA;
}

int ldpc_train_backward(ldpc_t* h, int32_t frames, int32_t iters, const float* alpha,
                        const float* beta, const float* grad_soft, int32_t soft_every,
                        float* grad_alpha, float* grad_beta, void* work, uint64_t work_bytes) {
    HandleView v;
    if (handle_view(h, &v) != LDPC_OK || !grad_soft || !grad_alpha || !grad_beta)
        return LDPC_ERR_BAD_POINTER;
    int rc = check_common(v, frames, iters, alpha, beta, work, work_bytes);
    if (rc != LDPC_OK) return rc;
    TrainWork w;
    const bool pk = packed_signs(v);
    carve(v.M, v.N, v.E, frames, iters, pk, (char*)work, &w);
    const LwArgs a = make_args(v, w.Fp, alpha, beta);
    cudaStream_t st = v.stream;
    // r and s hold the sums of this many iterations at least (of one in any case: there are no
    // more classes than bits)
    w.gsum = (double*)(((uintptr_t)w.r + 7) & ~(uintptr_t)7);
    const int64_t per = (2 * (int64_t)v.N * w.Fp * 4 - 8) / (16 * a.C);
    w.g0 = iters;
    const dim3 gi((v.N + 31) / 32, w.Fp / 32), bi(32, 8);
    const size_t plane = (size_t)frames * v.N;
    // ds^T = the loss gradient of the last posteriors
    k_lw_in<<<gi, bi, 0, st>>>(grad_soft + (soft_every ? (size_t)(iters - 1) * plane : 0), frames,
                               v.N, w.ds, w.Fp);
    const int V = lane_frames(v.M, w.Fp, v.num_sms, work), D = v.dg->ell_D;
    int launches = 1, g_top = iters;
    for (int t = iters; t >= 1; t--) {
        auto step = V == 4   ? (D == 8 ? launch_bwd<4, 8> : D == 16 ? launch_bwd<4, 16> : launch_bwd<4, 0>)
                    : V == 2 ? (D == 8 ? launch_bwd<2, 8> : D == 16 ? launch_bwd<2, 16> : launch_bwd<2, 0>)
                             : (D == 8 ? launch_bwd<1, 8> : D == 16 ? launch_bwd<1, 16> : launch_bwd<1, 0>);
        if (t == w.g0) {  // the sums of the next iterations
            w.g0 = (int32_t)std::max<int64_t>(0, t - per);
            if (cudaMemsetAsync(w.gsum, 0, (size_t)(t - w.g0) * a.C * 16, st) != cudaSuccess) return LDPC_ERR_CUDA;
            g_top = t;
        }
        step(a, w, t, t == iters, v.num_sms, soft_every && t > 1 ? grad_soft + (size_t)(t - 2) * plane : nullptr,
             frames, st);
        launches += t > 1 ? 2 : 1;
        if (t - 1 == w.g0) {
            const int n = (g_top - w.g0) * a.C;
            const size_t o = (size_t)w.g0 * a.C;
            k_lw_grad<<<(n + 127) / 128, 128, 0, st>>>(w.gsum, grad_alpha + o, grad_beta + o, n);
            launches++;
        }
    }
    *v.last_launches = launches;
    return cudaGetLastError() == cudaSuccess ? LDPC_OK : LDPC_ERR_CUDA;
}

}  // extern "C"
