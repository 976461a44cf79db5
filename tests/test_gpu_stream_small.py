"""GPU tests of the streaming variant on few frames (one or two frames a lane, register
kernels) around the sizes where the launch rule changes, on rows of at most 8, 16, 32 and of
more edges, in both modes, against the oracle; learned weights; infinite channel values, which
must give what the staged kernels give."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def code_of(rows):
    if rows == "8":
        return inputs.cfg_regular_576()
    if rows == "16":
        return inputs.irregular_code(480, 120, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 9)
    if rows == "32":
        return inputs.irregular_code(600, 100, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 9)
    return inputs.irregular_code(600, 50, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 9)


def decoder(code, mode, staged=False):
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    dec = Decoder.from_code(code, mode=mode)
    dec.set_variant("stream")
    if staged:
        dec.set_stream_staging(8, 2)
    return dec


@pytest.mark.parametrize("mode", ["fp32", "fixed"])
@pytest.mark.parametrize("rows", ["8", "16", "32", "40"])
def test_few_frames_match_oracle(mode, rows):
    import torch
    code = code_of(rows)
    assert {"8": 8, "16": 16, "32": 32, "40": 99}[rows] >= code.row_weights().max() > {"8": 2, "16": 8, "32": 16, "40": 32}[rows]
    g = oracle.Graph.from_code(code)
    dec = decoder(code, mode)
    for F in (1, 32, 33, 64, 65, 128, 129):
        llr = inputs.all_zero_awgn_llr(F, code.N, 4.5, code.design_rate, F)
        llr[0, : code.N // 4] *= -1.0  # one frame that does not stop
        for early_stop in (True, False):
            bits, it, ok, soft = dec.decode(torch.from_numpy(llr).cuda(), 9, early_stop=early_stop,
                                            check_every=2 if F == 33 else 1, want_ok=True, want_soft=True)
            kw = dict(early_stop=early_stop, check_every=2 if F == 33 else 1)
            want = (oracle.decode_f32(g, llr, 9, **kw) if mode == "fp32"
                    else oracle.decode_fixed(g, oracle.quantize(llr), 9, **kw))
            tag = (rows, mode, F, early_stop)
            assert (bits.cpu().numpy() == want[0]).all() and (it.cpu().numpy() == want[1]).all(), tag
            assert (ok.cpu().numpy() == want[2]).all(), tag
            s = want[3] if mode == "fp32" else want[3] * 0.25
            assert (soft.cpu().numpy() == s).all(), tag
    dec.close()


@pytest.mark.parametrize("rows", ["8", "32", "40"])
def test_few_frames_with_learned_weights(rows):
    import torch
    code = code_of(rows)
    cls, degrees = oracle.column_classes(code)
    rng = np.random.default_rng(4)
    a = rng.uniform(0.6, 1.0, (4, len(degrees))).astype(np.float32)
    b = rng.uniform(0.0, 0.3, (4, len(degrees))).astype(np.float32)
    g = oracle.Graph.from_code(code)
    dec = decoder(code, "fp32")
    dec.set_weights(a, b)
    for F in (7, 50):
        llr = inputs.all_zero_awgn_llr(F, code.N, 3.0, code.design_rate, F)
        bits, it, ok, soft = dec.decode(torch.from_numpy(llr).cuda(), 8, want_ok=True, want_soft=True)
        want = oracle.decode_weighted_f32(g, llr, 8, cls, a, b)
        assert (bits.cpu().numpy() == want[0]).all() and (it.cpu().numpy() == want[1]).all()
        assert (ok.cpu().numpy() == want[2]).all() and (soft.cpu().numpy() == want[3]).all()
    dec.close()


@pytest.mark.parametrize("conflicts", [False, True])
@pytest.mark.parametrize("rows", ["8", "16"])
def test_infinite_channel_values(rows, conflicts):
    """Known bits (infinite LLRs), down to rows with at most one finite value, whose second
    minimum is infinite: the narrow lanes agree with the staged kernels. With conflicts some
    are known wrongly, and infinities of both signs meet in a sum (NaN)."""
    import torch
    code = code_of(rows)
    llr = inputs.all_zero_awgn_llr(40, code.N, 2.0, code.design_rate, 3)
    rng = np.random.default_rng(8)
    for f in range(40):
        llr[f, rng.random(code.N) < f / 40.0] = np.inf
        if conflicts:
            llr[f, rng.random(code.N) < 0.1] *= -1.0
    x = torch.from_numpy(llr).cuda()
    got = []
    for staged in (False, True):
        dec = decoder(code, "fp32", staged)
        got.append(dec.decode(x, 6, early_stop=False, want_ok=True, want_soft=True))
        torch.cuda.synchronize()
        dec.close()
    for u, v in zip(*got):
        assert torch.equal(u.isnan(), v.isnan()) and torch.equal(torch.nan_to_num(u.float(), 7.0), torch.nan_to_num(v.float(), 7.0))
    assert bool(got[0][3].isinf().any())
