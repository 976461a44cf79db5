"""GPU tests of the early-stop resident decode where a CTA's rule on refilling ended slots
changes within a batch: stretches of frames that stop within an iteration of each other (no
refill: whole tiles), stretches whose iterations differ widely (slots refilled, the ones left
empty by then too), in both orders, against the oracle on every frame."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp32", "fixed"])
@pytest.mark.parametrize("check_every", [1, 3])
def test_rule_changes_within_a_batch(mode, check_every):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    code = inputs.regular_code(120, 60, 3, 6, 3)
    dec = Decoder.from_code(code, mode=mode)
    g = oracle.Graph.from_code(code)
    quiet = inputs.all_zero_awgn_llr(24001, code.N, 8.0, code.design_rate, 1)
    wide = inputs.all_zero_awgn_llr(24002, code.N, 2.0, code.design_rate, 2)
    for parts in ((quiet, wide, quiet), (wide, quiet, wide)):
        llr = np.concatenate(parts)
        got = dec.decode(torch.from_numpy(llr).cuda(), 12, check_every=check_every, want_ok=True, want_soft=True)
        kw = dict(early_stop=True, check_every=check_every)
        want = (oracle.decode_f32(g, llr, 12, **kw) if mode == "fp32"
                else oracle.decode_fixed(g, oracle.quantize(llr), 12, **kw))
        bits, it, ok, soft = (x.cpu().numpy() for x in got)
        assert (bits == want[0]).all() and (it == want[1]).all() and (ok == want[2]).all()
        assert (soft == (want[3] if mode == "fp32" else want[3] * 0.25)).all()
    dec.close()
