"""GPU tests of the streaming variant on full frame blocks with automatic staging: compressed
messages in the register check pass (FP32, padded rows of 8 and 16 slots and rows of up to 27
edges) and the register kernels beyond, around the longest row of each and the frame counts of
a block, in both modes, against the oracle; learned weights; the
messages read back; frame compaction; infinite channel values, whatever the message format."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def code_of(rows):
    if rows == "mixed":  # rows of 2 to 27 edges
        rng = np.random.default_rng(5)
        deg = np.concatenate([np.arange(2, 28), rng.integers(14, 28, 30)])
        r = np.repeat(np.arange(len(deg)), deg)
        c = 7 * np.arange(deg.sum()) % 180
        return inputs._make_code(len(deg), 180, r, c, "rows of 2 to 27 edges")
    N, M = {"8": (480, 204), "9": (480, 190), "16": (480, 102), "17": (500, 100), "21": (601, 100), "27": (540, 70), "28": (560, 69), "32": (640, 70)}[rows]
    return inputs.irregular_code(N, M, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 9)


def decoder(code, mode, compressed=True):
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    dec = Decoder.from_code(code, mode=mode)
    dec.set_variant("stream")
    dec.set_stream_messages(compressed)
    return dec


@pytest.mark.parametrize("mode", ["fp32", "fixed"])
@pytest.mark.parametrize("rows", ["mixed", "8", "9", "16", "17", "21", "27", "28", "32"])
def test_long_rows_match_oracle(mode, rows):
    import torch
    code = code_of(rows)
    longest = int(code.row_weights().max())
    assert longest == (27 if rows == "mixed" else int(rows))
    g = oracle.Graph.from_code(code)
    dec = decoder(code, mode)
    assert dec.stream_messages_compressed() == (mode == "fp32" and longest <= 27)
    for F in (65, 128, 257, 700):
        llr = inputs.all_zero_awgn_llr(F, code.N, 4.5, code.design_rate, F)
        llr[: F // 3, : code.N // 4] *= -1.0  # frames that do not stop (the others are compacted away)
        for early_stop in (True, False):
            kw = dict(early_stop=early_stop, check_every=2 if F == 257 else 1)
            bits, it, ok, soft = dec.decode(torch.from_numpy(llr).cuda(), 10, want_ok=True, want_soft=True, **kw)
            want = (oracle.decode_f32(g, llr, 10, **kw) if mode == "fp32"
                    else oracle.decode_fixed(g, oracle.quantize(llr), 10, **kw))
            tag = (rows, mode, F, early_stop)
            assert (bits.cpu().numpy() == want[0]).all() and (it.cpu().numpy() == want[1]).all(), tag
            assert (ok.cpu().numpy() == want[2]).all(), tag
            s = want[3] if mode == "fp32" else want[3] * 0.25
            assert (soft.cpu().numpy() == s).all(), tag
    dec.close()


@pytest.mark.parametrize("rows", ["mixed", "8", "16", "21", "32"])
def test_long_rows_with_learned_weights(rows):
    import torch
    code = code_of(rows)
    cls, degrees = oracle.column_classes(code)
    rng = np.random.default_rng(4)
    a = rng.uniform(0.6, 1.0, (4, len(degrees))).astype(np.float32)
    b = rng.uniform(0.0, 0.3, (4, len(degrees))).astype(np.float32)
    g = oracle.Graph.from_code(code)
    for compressed in (True, False):
        dec = decoder(code, "fp32", compressed)
        dec.set_weights(a, b)
        llr = inputs.all_zero_awgn_llr(150, code.N, 3.0, code.design_rate, 7)
        bits, it, ok, soft = dec.decode(torch.from_numpy(llr).cuda(), 8, want_ok=True, want_soft=True)
        want = oracle.decode_weighted_f32(g, llr, 8, cls, a, b)
        assert (bits.cpu().numpy() == want[0]).all() and (it.cpu().numpy() == want[1]).all()
        assert (ok.cpu().numpy() == want[2]).all() and (soft.cpu().numpy() == want[3]).all()
        dec.close()


@pytest.mark.parametrize("rows", ["8", "16", "27"])
def test_long_rows_messages_read_back(rows):
    import torch
    code = code_of(rows)
    llr = inputs.all_zero_awgn_llr(130, code.N, 4.0, code.design_rate, 2)
    g = oracle.Graph.from_code(code)
    dec = decoder(code, "fp32")
    for k in (1, 4):
        dec.decode(torch.from_numpy(llr).cuda(), k, early_stop=False)
        eta = dec.read_messages(130).cpu().numpy()
        for f in (0, 129):
            assert (eta[f] == oracle.trace_f32(g, llr[f], k)[3][k - 1]).all(), (k, f)
    dec.close()


@pytest.mark.parametrize("conflicts", [False, True])
@pytest.mark.parametrize("rows", ["mixed", "8", "16", "21"])
def test_infinite_channel_values(rows, conflicts):
    """Known bits, down to rows whose second minimum is infinite; with conflicts infinities of
    both signs meet in a sum (NaN). The register check pass gives what the staged one gives on
    padded rows, and what per-edge messages give on longer ones."""
    import torch
    code = code_of(rows)
    llr = inputs.all_zero_awgn_llr(140, code.N, 2.0, code.design_rate, 3)
    rng = np.random.default_rng(8)
    for f in range(140):
        llr[f, rng.random(code.N) < f / 140.0] = np.inf
        if conflicts:
            llr[f, rng.random(code.N) < 0.1] *= -1.0
    got = []
    padded = rows in ("8", "16")
    for reference in (True, False):
        dec = decoder(code, "fp32", compressed=padded or not reference)
        if padded and reference:
            dec.set_stream_staging(8, 2)
        assert dec.stream_messages_compressed() == (padded or not reference)
        got.append(dec.decode(torch.from_numpy(llr).cuda(), 6, early_stop=False, want_ok=True, want_soft=True))
        torch.cuda.synchronize()
        dec.close()
    for u, v in zip(*got):
        assert torch.equal(u.isnan(), v.isnan())
        assert torch.equal(torch.nan_to_num(u.float(), 7.0), torch.nan_to_num(v.float(), 7.0))
    assert bool(got[0][3].isinf().any())
