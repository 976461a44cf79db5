"""GPU tests of the resident launch plans that follow the batch size: narrow tiles for few
frames, two frames with the index arrays in global memory for codes that leave room for one.
Batches around the limits (one tile per multiprocessor, what runs at once), with and without
early stop, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def codes():
    return {"576": (inputs.cfg_regular_576(), 2.5),
            "2304": (inputs.cfg_qc_2304(), 4.0),
            # index arrays and one frame fit shared memory, with two frames the arrays do not:
            # in FP32 (short and long rows) and in fixed point
            "4096": (inputs.irregular_code(4096, 2048, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 304), 2.0),
            "5000": (inputs.irregular_code(5000, 1250, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 1), 3.5),
            "8192": (inputs.irregular_code(8192, 2731, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 305), 3.0)}


@pytest.mark.parametrize("mode", ["fp32", "fixed"])
@pytest.mark.parametrize("name", ["576", "2304", "4096", "5000", "8192"])
def test_batch_sizes_around_the_plan_limits(name, mode):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    code, snr = codes()[name]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = oracle.Graph.from_code(code)
    dec = Decoder.from_code(code, mode=mode)
    dec.set_variant("resident")
    top = 8 * sms + 1 if code.N < 2000 else 2 * sms + 1
    llr = inputs.all_zero_awgn_llr(top, code.N, snr, code.design_rate, 3)
    for es in (True, False):
        want = (oracle.decode_f32(g, llr, 9, early_stop=es) if mode == "fp32"
                else oracle.decode_fixed(g, oracle.quantize(llr), 9, early_stop=es))
        for F in sorted({1, sms, sms + 1, 2 * sms, 2 * sms + 1, min(top, 4 * sms + 1), top}):
            x = torch.from_numpy(llr[:F]).cuda()
            bits, it, ok, soft = dec.decode(x, 9, early_stop=es, want_ok=True, want_soft=True)
            tag = (name, mode, es, F)
            assert (bits.cpu().numpy() == want[0][:F]).all() and (it.cpu().numpy() == want[1][:F]).all(), tag
            assert (ok.cpu().numpy() == want[2][:F]).all(), tag
            s = want[3][:F] if mode == "fp32" else want[3][:F] * 0.25
            assert (soft.cpu().numpy() == s).all(), tag
    dec.close()
