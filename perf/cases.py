"""Performance cases of the Min-Sum decoder: what a user of this framework has it compute.

Every case goes through the public entry points (``Decoder.decode``, ``Batch``,
``WeightedMinSum``) with their default settings, on the codes of ``inputs.py``: single
frames, where latency counts, ordinary batches, the largest ones; codes whose frames stay
in shared memory and codes that stream; binary32 and fixed point; early stop on and off;
plain and learned Min-Sum; decoding and training (forward and backward).

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` /
``run`` execute one, ``work`` counts the bytes and operations one pass cannot do without and
``exact`` gives the computed outputs in 64 bits (the decisions, iteration counts and status
are whole numbers and have no such value).
"""
import functools
import math

import numpy as np
import torch

from paper_2507_10424_gb300 import inputs
from paper_2507_10424_gb300.ldpc import Batch, Decoder
from paper_2507_10424_gb300.learn import FrameSource, WeightedMinSum

# ------------------------------------------------------------------------------ cases


def _decode(**kw):
    case = dict(op="decode", mode="fp32", llr="f32", early_stop=True, check_every=1, soft=False,
                learned=False, code_seed=1)
    case.update(kw)
    return case


def listed():
    return [
        # One received word as it arrives: the latency of a call. (3,6) code, 2.5 dB.
        _decode(name="regular576_1f", code="regular", N=576, M=288, frames=1, iters=20,
                snr_lo=2.5, snr_hi=2.5, mean_iters=6),
        # An ordinary batch of the same code, stopping frame by frame.
        _decode(name="regular576_1024f", code="regular", N=576, M=288, frames=1024, iters=20,
                snr_lo=2.5, snr_hi=2.5, mean_iters=6),
        # Throughput decoding with a fixed number of iterations: the quasi-cyclic code on the
        # benchmark's batch.
        _decode(name="qc2304_65536f", code="qc", N=2304, M=1152, code_seed=2, frames=65536,
                iters=10, early_stop=False, snr_lo=1.0, snr_hi=3.0, mean_iters=10),
        # Fixed point on already quantised channel values, around the code's waterfall, an odd
        # number of frames: a receiver's inner loop.
        _decode(name="qc2304_fixed_i8_8191f", code="qc", N=2304, M=1152, code_seed=2,
                frames=8191, iters=20, mode="fixed", llr="i8", snr_lo=3.5, snr_hi=4.5, mean_iters=8),
        # The paper's protocol (200 frames, at most 60 iterations, the syndrome every 6) on the
        # code of its dimensions.
        _decode(name="paper8176_200f", code="paper", N=8176, M=1022, code_seed=4, frames=200,
                iters=60, check_every=6, snr_lo=3.0, snr_hi=3.6, mean_iters=58),
        # The large irregular code, every frame through all 50 iterations: the largest call.
        _decode(name="irregular64800_4096f", code="irregular238", N=64800, M=32400, code_seed=5,
                frames=4096, iters=50, early_stop=False, snr_lo=1.0, snr_hi=1.0, mean_iters=50),
        # The same code in fixed point at its waterfall, with early stop and soft output.
        _decode(name="irregular64800_fixed_1000f", code="irregular238", N=64800, M=32400,
                code_seed=5, frames=1000, iters=50, mode="fixed", snr_lo=1.4, snr_hi=1.4,
                mean_iters=40, soft=True),
        # Learned weights on the same code (three weight classes, 20 trained iterations).
        _decode(name="irr64800_learned_1024f", code="irregular238", N=64800, M=32400,
                code_seed=5, frames=1024, iters=40, snr_lo=1.2, snr_hi=1.4, mean_iters=36,
                learned=True),
        # A high-rate code with long rows (20 and 21 edges) that does not fit on chip, with
        # soft output: one of the mixed codes, as a call of its own.
        _decode(name="irregular16200_2001f", code="irregular2348", N=16200, M=2700, code_seed=307,
                frames=2001, iters=25, early_stop=False, snr_lo=2.0, snr_hi=2.0, mean_iters=25,
                soft=True),
        # One training step of the learned decoder, posteriors of every iteration: the small
        # code at its training batch size, and the large code.
        dict(name="train576_4096f", op="train", code="regular", N=576, M=288, code_seed=1,
             frames=4096, iters=10, snr_lo=1.0, snr_hi=4.0),
        dict(name="train64800_256f", op="train", code="irregular238", N=64800, M=32400,
             code_seed=5, frames=256, iters=20, snr_lo=0.8, snr_hi=1.4),
        # A server with several codes in use at once and few frames of each: one captured graph.
        dict(name="mixed8_64f", op="batch", codes=8, frames=64, iters=25, snr_lo=2.0,
             snr_hi=2.0, mean_iters=18),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Edge-frame-iterations of one drawn decode / training step at most (the largest listed
# decode has 4.1e10, the largest training step 1.0e9).
_MAX_DECODE, _MAX_TRAIN = 4.0e9, 4.0e8


def _draw_code(rng, large):
    """A code of the listed families: (kind, N, M, edges)."""
    if large:  # frames do not fit on chip: they stream
        if rng.random() < 0.5:
            N = 8 * _log_int(rng, 3000, 8100)
            return "irregular238", N, N // 2, int(3.125 * N)
        N = _log_int(rng, 12000, 24000)
        M = int(round(N * (1 - rng.choice(inputs.MIXED_RATES))))
        return "irregular2348", N, M, int(3.4 * N)
    kind = rng.choice(["regular", "qc", "irregular2348"])
    if kind == "regular":
        N = 2 * _log_int(rng, 60, 2000)
        return kind, N, N // 2, 3 * N
    if kind == "qc":
        N = 24 * _log_int(rng, 11, 96)
        return kind, N, N // 2, int(6.4 * N)
    N = _log_int(rng, 256, 8192)
    M = int(round(N * (1 - rng.choice(inputs.MIXED_RATES))))
    return kind, N, M, int(3.4 * N)


def draw(rng):
    """One more case of the listed ranges (rng: a random.Random), without a name."""
    what = rng.choice(["small", "small", "small", "large", "large", "learned", "train", "batch"])
    if what == "batch":
        return dict(op="batch", codes=rng.randint(2, 8), frames=_log_int(rng, 8, 300),
                    iters=rng.randint(5, 30), snr_lo=2.0, snr_hi=2.0, mean_iters=15)
    large = what == "large" or (what != "small" and rng.random() < 0.4)
    kind, N, M, E = _draw_code(rng, large)
    seed = rng.randint(1, 1 << 20)
    if what == "train":
        T = rng.randint(4, 20)
        cap = max(1, min(4096, int(_MAX_TRAIN / (E * T))))
        return dict(op="train", code=kind, N=N, M=M, code_seed=seed, frames=_log_int(rng, 1, cap),
                    iters=T, snr_lo=1.0, snr_hi=4.0)
    iters = rng.randint(5, 60)
    cap = max(1, min(4096 if large else 65536, int(_MAX_DECODE / (E * iters))))
    fixed = what != "learned" and rng.random() < 0.5
    es = rng.random() < 0.7
    lo = rng.uniform(1.0, 4.0)
    return _decode(code=kind, N=N, M=M, code_seed=seed, frames=_log_int(rng, 1, cap), iters=iters,
                   mode="fixed" if fixed else "fp32",
                   llr="i8" if fixed and rng.random() < 0.5 else "f32",
                   early_stop=es, check_every=rng.choice([1, 1, 1, 2, 6]), soft=rng.random() < 0.4,
                   learned=what == "learned", snr_lo=lo, snr_hi=lo + rng.uniform(0.0, 1.5),
                   mean_iters=max(1, iters // 2) if es else iters)


# ------------------------------------------------------------------- codes and channel


@functools.lru_cache(maxsize=64)
def _code(kind, N, M, seed):
    if kind == "regular":
        return inputs.regular_code(N, M, 3, 6, seed)
    if kind == "qc":
        return inputs.qc_code(12, 24, N // 24, 0.5, seed)
    if kind == "paper":
        return inputs.cfg_paper_shaped(seed)
    if kind == "irregular238":
        return inputs.irregular_code(N, M, [2, 3, 8], [0.5, 0.375, 0.125], seed)
    return inputs.irregular_code(N, M, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], seed)


@functools.lru_cache(maxsize=1)
def _mixed():
    return inputs.cfg_mixed_codes()[0]


@functools.lru_cache(maxsize=64)
def _source(kind, N, M, seed):
    """Frames of a code: random codewords where the GF(2) encoder is practical, else the
    all-zero codeword (Min-Sum is symmetric in the codeword sent)."""
    code = _code(kind, N, M, seed)
    return FrameSource(code, encode=N <= 2304)


def _key(case):
    return case["code"], case["N"], case["M"], case["code_seed"]


def _frames(case, seed):
    """(llr float32 [F][N], bits uint8 [F][N]) on the GPU, from the seed alone."""
    src = _source(*_key(case))
    src.gen.manual_seed(seed)
    return src.batch(case["frames"], (case["snr_lo"], case["snr_hi"]))


def _llr(case, seed):
    """The channel values of a decode: binary32, or already quantised to int8 steps of 1/4."""
    llr, _ = _frames(case, seed)
    if case["llr"] == "i8":
        return torch.clamp(torch.round(4.0 * llr), -127, 127).to(torch.int8)
    return llr


def _weights(classes, iters):
    """Weights as training leaves them: alpha rises and beta falls over the iterations, the
    classes a little apart. float32 [iters][classes]."""
    t = np.linspace(0.0, 1.0, max(iters, 2))[:iters, None]
    c = 0.01 * np.arange(classes)[None, :]
    alpha = 0.74 + 0.18 * t + c
    beta = 0.21 - 0.10 * t + 0.5 * c
    return alpha.astype(np.float32), beta.astype(np.float32)


def _n_classes(code):
    return len(np.unique(code.col_weights()))


def _batch_llrs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out = []
    for code in _mixed()[:case["codes"]]:
        s2 = inputs.noise_sigma2(case["snr_lo"], code.design_rate)
        y = 1.0 + math.sqrt(s2) * torch.randn((case["frames"], code.N), generator=gen, device="cuda")
        out.append(2.0 / s2 * y)
    return out


def _train_inputs(case, seed):
    """(llr, alpha, beta, grad): a batch, weights near the trained ones, and the gradient of
    the mean cross-entropy with respect to every iteration's posteriors, taken at the channel
    values."""
    llr, bits = _frames(case, seed)
    T = case["iters"]
    a, b = _weights(_n_classes(_code(*_key(case))), T)
    g = (bits.float() - torch.sigmoid(-llr)) / (T * llr.numel())
    ramp = torch.linspace(1.0, 0.6, T, device="cuda").view(T, 1, 1)
    return llr, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), g.unsqueeze(0) * ramp


# ------------------------------------------------------------------------ prepare, run


def prepare(case, seed):
    if case["op"] == "batch":
        batch = Batch([Decoder.from_code(c) for c in _mixed()[:case["codes"]]])
        outs = [batch.set_io(k, llr, want_ok=True) for k, llr in enumerate(_batch_llrs(case, seed))]
        torch.cuda.synchronize()  # the inputs are ready before the batch's own stream uses them
        batch.prepare(case["iters"])
        batch.capture()
        return dict(op="batch", batch=batch, outs=[o[:3] for o in outs])
    code = _code(*_key(case))
    if case["op"] == "train":
        llr, alpha, beta, grad = _train_inputs(case, seed)
        return dict(op="train", dec=Decoder.from_code(code), llr=llr, alpha=alpha.requires_grad_(),
                    beta=beta.requires_grad_(), grad=grad)
    dec = Decoder.from_code(code, mode=case["mode"])
    if case["learned"]:
        dec.set_weights(*_weights(len(dec.classes()), 20))
    return dict(op="decode", dec=dec, llr=_llr(case, seed), iters=case["iters"],
                early_stop=case["early_stop"], check_every=case["check_every"], soft=case["soft"])


def run(state):
    if state["op"] == "batch":
        # the graph runs on the batch's own stream, ordered with the caller's
        batch, cur = state["batch"], torch.cuda.current_stream()
        batch.stream.wait_stream(cur)
        batch.replay()
        cur.wait_stream(batch.stream)
        return state["outs"]
    if state["op"] == "train":
        soft = WeightedMinSum.apply(state["dec"], state["llr"], state["alpha"], state["beta"], True)
        ga, gb = torch.autograd.grad(soft, (state["alpha"], state["beta"]), state["grad"])
        return dict(soft=soft.detach(), grad_alpha=ga, grad_beta=gb)
    bits, iters, ok, soft = state["dec"].decode(
        state["llr"], state["iters"], early_stop=state["early_stop"],
        check_every=state["check_every"], want_ok=True, want_soft=state["soft"])
    out = dict(bits=bits, iters=iters, ok=ok)
    if soft is not None:
        out["soft"] = soft
    return out


# -------------------------------------------------------------------------------- work


def work(case):
    """Bytes: each input read once, each output written once. Operations per edge, frame and
    iteration: check update (difference, magnitude, two minima, sign, pick) and the column
    sum, 7; the adjoint takes about as many again."""
    F = case["frames"]
    if case["op"] == "batch":
        codes = _mixed()[:case["codes"]]
        return dict(bytes=float(sum(F * (5 * c.N + 5) for c in codes)),
                    flops=float(sum(7 * c.E * F * case["mean_iters"] for c in codes)))
    code = _code(*_key(case))
    N, E = code.N, code.E
    if case["op"] == "train":
        T = case["iters"]
        return dict(bytes=float(4 * F * N * (1 + 2 * T)), flops=float(14 * E * F * T))
    per_bit = (1 if case["llr"] == "i8" else 4) + 1 + (4 if case["soft"] else 0)
    return dict(bytes=float(F * (N * per_bit + 5)), flops=float(7 * E * F * case["mean_iters"]))


# ------------------------------------------------------------------------------- exact


def _padded(code):
    """(columns of each check, padded with N; slots of each bit's edges, padded with M D)."""
    rp, ci = code.csr()
    deg = np.diff(rp)
    D = int(deg.max())
    slot = np.repeat(np.arange(code.M) * D, deg) + np.arange(code.E) - np.repeat(rp[:-1], deg)
    cols = np.full(code.M * D, code.N, np.int64)
    cols[slot] = ci
    order = np.argsort(ci, kind="stable")
    cdeg = code.col_weights()
    start = np.concatenate([[0], np.cumsum(cdeg)[:-1]])
    slots = np.full((code.N, int(cdeg.max())), code.M * D, np.int64)
    slots[np.repeat(np.arange(code.N), cdeg), np.arange(code.E) - np.repeat(start, cdeg)] = slot[order]
    return torch.from_numpy(cols).cuda(), torch.from_numpy(slots).cuda(), D


def _check_pick(lam, D, M):
    """(positions of the smallest and second smallest magnitude, extrinsic signs) of each
    check; lam [M][D][F], padding +inf."""
    mag = lam.abs()
    i0 = mag.argmin(1, keepdim=True)
    i1 = mag.scatter(1, i0, math.inf).argmin(1, keepdim=True)
    neg = lam < 0
    sign = torch.where(neg ^ (neg.sum(1, keepdim=True) % 2 == 1), -1.0, 1.0).to(lam.dtype)
    return i0, i1, sign


def _col_sum(eta, slots):
    """Sum of each bit's messages; eta [M D][F]."""
    ext = torch.cat([eta, torch.zeros_like(eta[:1])])
    out = torch.zeros((slots.shape[0], eta.shape[1]), dtype=eta.dtype, device=eta.device)
    for k in range(slots.shape[1]):
        out = out + ext[slots[:, k]]
    return out


def _posteriors64(case, code, llr):
    """Posteriors [F][N] of a decode of these frames in 64-bit arithmetic (fixed point: whole
    quarter steps with the mode's saturation, exact)."""
    M, N = code.M, code.N
    cols, slots, D = _padded(code)
    fixed = case["mode"] == "fixed"
    r = llr.double().T.contiguous()
    if fixed and case["llr"] == "f32":
        r = torch.clamp(torch.round(4.0 * r), -127.0, 127.0)
    F = r.shape[1]
    pos = torch.arange(D, device="cuda").view(1, D, 1)
    if case["learned"]:
        wa, wb = _weights(_n_classes(code), 20)
        cls = np.searchsorted(np.unique(code.col_weights()), code.col_weights())
        cls = torch.from_numpy(np.append(cls, 0)).cuda()[cols]
    s, eta = r.clone(), torch.zeros((M * D, F), dtype=torch.float64, device="cuda")
    run_f = torch.ones(F, dtype=torch.bool, device="cuda")
    for k in range(1, case["iters"] + 1):
        if case["early_stop"] and (k - 1) % case["check_every"] == 0:
            hard = torch.cat([s < 0, torch.zeros((1, F), dtype=torch.bool, device="cuda")])
            run_f &= (hard[cols].view(M, D, F).sum(1) % 2).any(0)
            if not bool(run_f.any()):
                break
        lam = torch.cat([s, torch.full((1, F), math.inf, dtype=s.dtype, device="cuda")])[cols] - eta
        if fixed:
            lam = torch.where(lam == math.inf, lam, lam.clamp(-32767, 32767))
        lam = lam.view(M, D, F)
        i0, i1, sign = _check_pick(lam, D, M)
        m0, m1 = lam.gather(1, i0).abs(), lam.gather(1, i1).abs()
        m = torch.where(pos == i0, m1, m0)
        if case["learned"]:
            row = min(k, 20) - 1
            a = torch.from_numpy(wa[row]).double().cuda()[cls].view(M, D, 1)
            b = torch.from_numpy(wb[row]).double().cuda()[cls].view(M, D, 1)
            m = torch.clamp(a * m - b, min=0.0)
        eta = (m * sign).view(M * D, F)
        new = r + _col_sum(eta, slots)
        if fixed:
            new = new.clamp(-32767, 32767)
        s = torch.where(run_f, new, s)
    return (0.25 * s if fixed else s).T.contiguous()


def _train64(case, code, llr, alpha, beta, grad):
    """(soft [T][F][N], gradient of the weights) of these frames by autograd in 64 bits."""
    M, T, F = code.M, case["iters"], llr.shape[0]
    cols, slots, D = _padded(code)
    cls = np.searchsorted(np.unique(code.col_weights()), code.col_weights())
    cls = torch.from_numpy(np.append(cls, 0)).cuda()[cols]
    a = alpha.detach().double().requires_grad_()
    b = beta.detach().double().requires_grad_()
    pos = torch.arange(D, device="cuda").view(1, D, 1)
    r = llr.double().T.contiguous()
    s, eta, soft = r, torch.zeros((M * D, F), dtype=torch.float64, device="cuda"), []
    for t in range(T):
        ext = torch.cat([s, torch.full((1, F), math.inf, dtype=s.dtype, device="cuda")])
        lam = (ext[cols] - eta).view(M, D, F)
        i0, i1, sign = _check_pick(lam.detach(), D, M)
        m0, m1 = lam.gather(1, i0).abs(), lam.gather(1, i1).abs()
        m = torch.where(pos == i0, m1, m0)
        w = torch.relu(a[t][cls].view(M, D, 1) * m - b[t][cls].view(M, D, 1))
        eta = (w * sign).view(M * D, F)
        s = r + _col_sum(eta, slots)
        soft.append(s.T)
    soft = torch.stack(soft)
    ga, gb = torch.autograd.grad(soft, (a, b), grad.double())
    return soft.detach(), ga, gb


# A frame that does not converge follows a chaotic path: past some tens of iterations the
# last bit of a binary32 sum decides its posteriors, and no 64-bit value stands for them.
_MAX_EXACT_ITERS = 25


def exact(case, seed):
    if case["op"] == "batch":
        return None
    code = _code(*_key(case))
    per_frame = 8 * code.M * int(code.row_weights().max())  # bytes of one edge array, 64 bits
    if case["op"] == "train":
        llr, alpha, beta, grad = _train_inputs(case, seed)
        step = max(1, int(2e10 / (per_frame * 8 * case["iters"])))
        soft = torch.empty((case["iters"],) + tuple(llr.shape), dtype=torch.float64, device="cuda")
        ga = torch.zeros(alpha.shape, dtype=torch.float64, device="cuda")
        gb = torch.zeros_like(ga)
        for f in range(0, case["frames"], step):
            o, x, y = _train64(case, code, llr[f:f + step], alpha, beta, grad[:, f:f + step])
            soft[:, f:f + step] = o
            ga += x
            gb += y
        return dict(soft=soft, grad_alpha=ga, grad_beta=gb)
    if not case["soft"] or (case["mode"] == "fp32" and case["iters"] > _MAX_EXACT_ITERS):
        return None
    llr = _llr(case, seed)
    step = max(1, int(4e9 / per_frame))
    soft = torch.cat([_posteriors64(case, code, llr[f:f + step]) for f in range(0, case["frames"], step)])
    return dict(bits=None, iters=None, ok=None, soft=soft)
