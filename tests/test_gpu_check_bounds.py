"""GPU tests of the check pass on compressed messages where warps take several rows and frame
blocks without running frames are skipped: batches of many blocks whose frames stop at
different iterations (compactions in between) or all at once, a last row group that is ragged,
rows of at most 8 and 16 edges, learned weights, every other iteration tested, against the
oracle on a sample of the frames; and batches of 65 to 128 frames, whose second block of the
frame stride is padding."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def check(code, llr, L, weights, sample, **kw):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    dec = Decoder.from_code(code)
    dec.set_variant("stream")
    g = oracle.Graph.from_code(code)
    cls, degrees = oracle.column_classes(code)
    if weights:
        rng = np.random.default_rng(4)
        a = rng.uniform(0.7, 1.0, (4, len(degrees))).astype(np.float32)
        b = rng.uniform(0.0, 0.1, (4, len(degrees))).astype(np.float32)
        dec.set_weights(a, b)
    got = [x.cpu().numpy()[sample] for x in dec.decode(torch.from_numpy(llr).cuda(), L, want_ok=True, want_soft=True, **kw)]
    x = llr[sample]
    want = oracle.decode_weighted_f32(g, x, L, cls, a, b, **kw) if weights else oracle.decode_f32(g, x, L, **kw)
    for name, u, v in zip(("bits", "iters", "ok", "soft"), got, want):
        assert (u == v).all(), name
    dec.close()
    return want[1]


@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("rows,check_every", [(8, 1), (8, 2), (16, 1)])
def test_blocks_that_stop(rows, check_every, weights):
    N, M = (1998, 999) if rows == 8 else (2001, 501)  # 999 and 501: no multiple of 16
    code = inputs.irregular_code(N, M, [2, 3, 8], [0.5, 0.375, 0.125], 9)
    assert (8 if rows == 16 else 2) < code.row_weights().max() <= rows
    F = 128 * 152 * 128 // M + 129  # frames: enough rows times blocks on GPUs of up to 152 SMs
    rate = code.design_rate
    sample = np.r_[0:4, F // 2:F // 2 + 6, F - 4:F]
    quiet = inputs.all_zero_awgn_llr(F, N, 7.0, rate, 1)  # all stop within a few iterations
    it = check(code, quiet, 30, weights, sample, check_every=check_every)
    assert it.max() < 12
    mixed = quiet.copy()  # the second half runs on, some to the limit
    mixed[F // 2:] = inputs.all_zero_awgn_llr(F - F // 2, N, 2.0 if rows == 8 else 3.5, rate, 2)
    it = check(code, mixed, 14, weights, sample, check_every=check_every)
    assert it.max() > 6 and it.min() < 6


@pytest.mark.parametrize("early_stop", [False, True])
@pytest.mark.parametrize("rows", [8, 16, 20])
@pytest.mark.parametrize("frames", [65, 128, 129])
def test_padding_blocks(rows, frames, early_stop):
    M = {8: 300, 16: 150, 20: 100}[rows]
    code = inputs.irregular_code(600, M, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 9)
    llr = inputs.all_zero_awgn_llr(frames, code.N, 4.0, code.design_rate, frames)
    check(code, llr, 8, False, np.arange(frames), early_stop=early_stop)
