"""GPU tests of ldpc_read_messages after calls that touch the handle between the decode and the
read: ldpc_reserve, which sets a frame stride of its own, and allocates a workspace of more
frames, against the oracle's messages; and ldpc_set_weights, which leaves the messages of the
decode as they were, in either format."""
import numpy as np
import pytest

import oracle
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def decoder(code, mode="fp32"):
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    dec = Decoder.from_code(code, mode=mode)
    dec.set_variant("stream")
    return dec


def code_of(rows):
    if rows == "6":
        return inputs.cfg_regular_576()
    return inputs.irregular_code(600, 100, [2, 3, 4, 8], [0.3, 0.4, 0.2, 0.1], 9)


@pytest.mark.parametrize("mode", ["fp32", "fixed"])
@pytest.mark.parametrize("rows", ["6", "20"])
@pytest.mark.parametrize("frames", [10, 33, 65, 300])
def test_messages_after_reserve(rows, mode, frames):
    import torch
    from paper_2507_10424_gb300 import ldpc
    code = code_of(rows)
    g = oracle.Graph.from_code(code)
    dec = decoder(code, mode)
    llr = inputs.all_zero_awgn_llr(frames, code.N, 2.0, code.design_rate, 3)
    x = torch.from_numpy(llr).cuda()
    dec.decode(x, 3, early_stop=False)
    for reserve in (0, 1, 100, frames):  # none of them needs a larger workspace
        dec.reserve(reserve)
        eta = dec.read_messages(frames).cpu().numpy()
        for f in (0, 1, frames - 1):
            if mode == "fp32":
                assert (eta[f] == oracle.trace_f32(g, llr[f], 3)[3][2]).all(), (reserve, f)
            else:
                assert (eta[f] * 4 == oracle.trace_fixed(g, oracle.quantize(llr[f]), 3)[3][2]).all(), (reserve, f)
    dec.reserve(2000)  # a new workspace: the messages are gone
    with pytest.raises(ldpc.LdpcError) as e:
        dec.read_messages(1)
    assert e.value.status == ldpc.LDPC_ERR_UNSUPPORTED
    dec.decode(x, 3, early_stop=False)
    assert torch.equal(dec.read_messages(frames).cpu(), torch.from_numpy(eta))
    dec.close()


@pytest.mark.parametrize("compressed", [True, False])
@pytest.mark.parametrize("rows", ["6", "20"])
def test_messages_after_set_weights(rows, compressed):
    import torch
    code = code_of(rows)
    C = len(oracle.column_classes(code)[1])
    rng = np.random.default_rng(4)
    tables = [(rng.uniform(0.6, 1.0, (3, C)).astype(np.float32), rng.uniform(0.0, 0.3, (3, C)).astype(np.float32))
              for _ in range(3)]
    x = torch.from_numpy(inputs.all_zero_awgn_llr(130, code.N, 2.0, code.design_rate, 3)).cuda()
    dec = decoder(code)
    dec.set_stream_messages(compressed)
    dec.decode(x, 2, early_stop=False)  # no weights
    plain = dec.read_messages(130).clone()
    dec.set_weights(*tables[0])
    assert torch.equal(dec.read_messages(130), plain)
    dec.decode(x, 2, early_stop=False)
    want = dec.read_messages(130).clone()
    assert not torch.equal(want, plain)
    for t in tables[1:]:
        dec.set_weights(*t)
        assert torch.equal(dec.read_messages(130), want)
    dec.set_weights(None, None)
    assert torch.equal(dec.read_messages(130), want)
    dec.decode(x, 2, early_stop=False)
    assert torch.equal(dec.read_messages(130), plain)
    dec.close()
