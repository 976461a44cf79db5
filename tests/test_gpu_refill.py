"""GPU tests of early-stop decodes with more frames than the resident kernel has slots: frames
stop at different iterations and give their slots to the next ones of the batch. Every output
against the oracle, bit for bit, over tile widths, index placements, both modes and input
types, cadences of the syndrome test and iteration limits."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def check(code, llr, mode, L, every, shape, i8=False):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder, LdpcError
    build.build()
    dec = Decoder.from_code(code, mode=mode)
    dec.set_variant("resident")
    try:
        dec.set_tuning(*shape)
    except LdpcError:
        pytest.skip(f"{shape} does not fit this code")
    x = oracle.quantize(llr) if i8 else llr
    bits, it, ok, soft = dec.decode(torch.from_numpy(x).cuda(), L, check_every=every, want_ok=True, want_soft=True)
    g = oracle.Graph.from_code(code)
    want = (oracle.decode_f32(g, llr, L, check_every=every) if mode == "fp32"
            else oracle.decode_fixed(g, oracle.quantize(llr), L, check_every=every))
    assert (it.cpu().numpy() == want[1]).all()
    assert (ok.cpu().numpy() == want[2]).all()
    assert (bits.cpu().numpy() == want[0]).all()
    assert (soft.cpu().numpy() == (want[3] if mode == "fp32" else want[3] * 0.25)).all()
    dec.close()
    return want[1]


@pytest.mark.parametrize("mode", ["fp32", "fixed"])
@pytest.mark.parametrize("shape", [(4, 288, 1), (2, 640, 1), (1, 1024, 1), (2, 96, 2), (1, 64, 2)])
def test_more_frames_than_slots(mode, shape):
    code = inputs.cfg_regular_576()
    llr = np.concatenate([inputs.all_zero_awgn_llr(1500, code.N, snr, code.design_rate, k)
                          for k, snr in enumerate((1.0, 2.5, 3.0, 6.0, 2.0, 3.5))])
    llr = llr[np.random.default_rng(3).permutation(len(llr))][:8999]
    for L, every in ((20, 1), (13, 3), (1, 1)):
        it = check(code, llr, mode, L, every, shape)
        assert L == 1 or len(np.unique(it)) > 3  # frames stop apart


@pytest.mark.parametrize("i8", [False, True])
def test_more_frames_than_slots_one_cta_a_multiprocessor(i8):
    code = inputs.cfg_qc_2304()
    llr = np.concatenate([inputs.all_zero_awgn_llr(300, code.N, snr, code.design_rate, k)
                          for k, snr in enumerate((3.0, 4.0, 4.5, 6.0, 4.2))])
    llr = llr[np.random.default_rng(3).permutation(len(llr))]
    check(code, llr, "fixed", 15, 1, (4, 768, 1), i8)
    if not i8:
        check(code, llr, "fp32", 15, 2, (2, 768, 1))
