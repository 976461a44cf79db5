"""GPU tests of what creating a handle leaves out: the search for a column order of a code that
streams in the handle's mode, which must not matter to the other mode, where the code stays on
chip; and bit-packed rows on either side of the size up to which they share the index arrays'
allocation."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_other_mode_of_a_streaming_code():
    import torch
    from paper_2507_10424_gb300 import build, ldpc
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    code = inputs.irregular_code(12288, 3072, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 6)
    g = oracle.Graph.from_code(code)
    llr = inputs.all_zero_awgn_llr(40, code.N, 3.2, code.design_rate, 3)
    x = torch.from_numpy(llr).cuda()
    dec = Decoder.from_code(code)
    assert dec.variant() == "stream"
    assert ldpc.ldpc_set_mode(dec.h, ldpc.LDPC_MODE_FIXED) == 0
    assert dec.variant() == "resident"
    want = oracle.decode_fixed(g, oracle.quantize(llr), 9)
    for d in (dec, Decoder.from_code(code, mode="fixed")):
        bits, it, ok, soft = (t.cpu().numpy() for t in d.decode(x, 9, want_ok=True, want_soft=True))
        assert (bits == want[0]).all() and (it == want[1]).all() and (ok == want[2]).all()
        assert (soft == want[3] * 0.25).all()
        d.close()


@pytest.mark.parametrize("N", [1440, 1536])  # words of N x N bits: below and above 2^16
def test_packed_rows_of_either_size(N):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    assert (N * (N // 32) < 1 << 16) == (N == 1440)
    code = inputs.regular_code(N, N // 2, 3, 6, 3)
    sets = [list(code.cols[code.rows == i] + 1) for i in range(code.M)] + [[] for _ in range(N - code.M)]
    code = inputs.code_from_index_sets(sets, N)  # rows without edges up to N rows
    llr = inputs.all_zero_awgn_llr(3, N, 2.0, 0.5, 3)
    dec = Decoder.from_code(code)
    dec.set_variant("dense")  # reads the packed rows
    bits, it, ok, _ = (t if t is None else t.cpu().numpy() for t in dec.decode(torch.from_numpy(llr).cuda(), 3, want_ok=True))
    want = oracle.decode_f32(oracle.Graph.from_code(code), llr, 3)
    assert (bits == want[0]).all() and (it == want[1]).all() and (ok == want[2]).all()
    dec.close()
