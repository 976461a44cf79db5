// Resident variant, host side: the launch plan (frames per tile, index placement,
// register budget of the row sweep, CTA size) and the decode entry used by the C ABI.
#include "resident.cuh"

namespace ldpc_impl {
using namespace resident;

ResidentPlan resident_plan(int mode, const DevGraph& dg, int32_t N, int device,
                           const ResidentTuning& tune, int w_entries) {
    ResidentPlan p;
    if (!dg.sliced) return p;
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    const int tb = mode == kModeFP32 ? 4 : 2;
    const size_t budget = (size_t)std::max(0, optin - 256);  // static shared memory
    // up to four interleaved frames (registers); index arrays in shared memory preferred
    const int fts[] = {4, 2, 1};
    for (int idx = 1; idx >= 0 && !p.ok; idx--)
        for (int ft : fts) {
            if ((tune.idx == 1 && !idx) || (tune.idx == 2 && idx)) continue;
            if (ft * tb > 16 || (!idx && ft > 2)) continue;
            if (tune.FT && ft != tune.FT) continue;
            const ResLayout L = res_layout(tb, ft, dg.E_pad, dg.Ec_pad, dg.n_rslices, dg.n_cslices, N, idx,
                                           mode == kModeFP32 ? w_entries : 0);
            if (L.total <= budget) {
                p.ok = 1;
                p.FT = ft;
                p.idx_smem = idx;
                p.smem = L.total;
                break;
            }
        }
    if (!p.ok) return p;
    int per_sm = 0;
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
    p.ctas_per_sm = std::max(1, (int)(per_sm / (p.smem + 1024)));  // as far as shared memory goes
    if (tune.threads) {
        if (tune.threads % 32 || tune.threads < 64 || tune.threads > kMaxThreads) return ResidentPlan();
        p.threads = tune.threads;
        return p;
    }
    // threads: balance latency hiding (resident warps per SM, counted up to 24) against
    // the padding of the last round of row and column tasks (rows weigh twice: two sweeps)
    const int ctas_smem = p.ctas_per_sm;
    const int rt = dg.n_rslices * 32;
    const double useful = 2.0 * rt + N;
    double best = -1.0;
    for (int t = 256; t <= kMaxThreads; t += 32) {
        const int ctas = std::min(ctas_smem, 2048 / t);
        const double warps = std::min(24.0, (double)ctas * t / 32.0);
        const double padded = 2.0 * ((rt + t - 1) / t) * t + (double)((N + t - 1) / t) * t;
        const double score = warps * useful / padded;
        if (score > best + 1e-9) {
            best = score;
            p.threads = t;
        }
    }
    return p;
}

// A batch that does not fill the GPU takes tiles of fewer frames: a tile's iteration takes
// longer the wider it is (one frame of FP32 on N=576: 21 us a decode against 26 us on 4-frame
// tiles), and with early stop fewer frames wait for the slowest of their tile. The limit is
// one tile per SM without early stop (N=576, 8 iterations, FP32, 1 / 2 / 4 frames per tile: 152
// frames 21.1 / 22.5 / 27.7 us, 1024 frames 38.7 / 38.4 / 34.2 us) and with early stop what
// runs at once (1024 frames, 20 iterations: 62.8 / 67.7 / 71.1 us; 4096 frames: 157 / 151 / 141
// us), four tiles per SM for pairs of FP32 frames (2048 frames: 94.7 / 97.6 / 95.8 us). Fixed
// point keeps its frames in packed pairs (QC N=2304, 304 frames, 8 iterations: 68.6 / 46.7 /
// 64.5 us).
int resident_narrow(int mode, int FT, const ResidentPlan narrow[2], int32_t frames, int early_stop, int num_sms) {
    for (int ft = mode == kModeFixed ? 2 : 1; ft < FT && ft <= 2; ft++) {
        const ResidentPlan& p = narrow[ft - 1];
        if (!p.ok || !p.idx_smem) continue;
        const int tiles = (frames + ft - 1) / ft;
        int per_sm = 1;
        if (early_stop) {
            per_sm = std::min(p.ctas_per_sm, 2048 / p.threads);
            if (mode == kModeFP32 && ft == 2) per_sm = std::min(per_sm, 4);
        }
        if (tiles <= num_sms * std::max(1, per_sm)) return ft;
    }
    return 0;
}

// A code whose index arrays leave room for one frame only: the room is better spent on a second
// frame, the index arrays then coming from L1 and L2, once there are more frames than SMs.
// Measured, 4096 frames, one frame / two frames, fixed point (whose packed arithmetic needs
// the pair): N=8192 8 iterations 1822 -> 1290 us, N=7000 with early stop 3293 -> 2163 us; FP32:
// N=4096 (rows of 6-7) 929 -> 764 us and with early stop 1832 -> 1591 us, N=5000 (rows of 13-14)
// 1162 -> 1070 us but with early stop 1198 -> 1257 us: the syndrome's gather then reads a
// position per edge from global memory, which long rows wait for.
bool resident_wide(int mode, const ResidentPlan& p, int32_t max_dc, int32_t frames, int early_stop, int num_sms) {
    return p.FT == 1 && p.idx_smem && frames > num_sms && (mode == kModeFixed || !early_stop || max_dc <= 8);
}

int resident_decode(int mode, const DevGraph& dg, const ResidentPlan& p, const DecodeArgs& a,
                    int32_t* tile_counter, int num_sms, cudaStream_t st) {
    ResArgs ra;
    ra.r_base = dg.r_base;
    ra.r_deg = dg.r_deg;
    ra.r_slot_pos = dg.r_slot_pos;
    ra.c_base = dg.c_base;
    ra.c_deg = dg.c_deg;
    ra.c_slot = dg.c_slot;
    ra.col_pos = dg.col_pos;
    ra.r_slot_cls = dg.r_slot_cls;
    ra.idx_blob = dg.idx_blob;
    ra.w_rows = mode == kModeFP32 ? a.w_rows : 0;
    ra.n_classes = a.n_classes;
    ra.w_alpha = a.w_alpha;
    ra.w_beta = a.w_beta;
    ra.n_rsl = dg.n_rslices;
    ra.n_csl = dg.n_cslices;
    ra.E_pad = dg.E_pad;
    ra.Ec_pad = dg.Ec_pad;
    ra.N = a.N;
    ra.llr = a.llr;
    ra.llr_i8 = a.llr_is_i8;
    ra.frames = a.frames;
    ra.n_tiles = (a.frames + p.FT - 1) / p.FT;
    ra.L = a.L;
    ra.early_stop = a.early_stop;
    ra.check_every = a.check_every;
    ra.paper = a.paper_slicer;
    ra.out_bits = a.out_bits;
    ra.out_iters = a.out_iters;
    ra.out_ok = a.out_ok;
    ra.out_soft = a.out_soft;
    ra.tile_counter = tile_counter;
    if (use_es(ra))
        return mode == kModeFP32 ? dispatch_fp32_es(ra, p, num_sms, st)
                                 : dispatch_fixed_es(ra, p, num_sms, st);
    return mode == kModeFP32 ? dispatch_fp32(ra, p, num_sms, st) : dispatch_fixed(ra, p, num_sms, st);
}

}  // namespace ldpc_impl
