"""GPU tests of the training kernels over the shapes their launch rules tell apart: 1, 2 and 4
frames a lane with ragged last lane groups, rows of at most 16 edges and longer ones, one weight
class, several, and more than the shared-memory accumulators hold; against the autograd
reference in 64 bits. The gradients are sums over the frames in binary32: 1e-3 of the largest
entry bounds their rounding and the frames whose minima tie within binary32."""
import ctypes

import numpy as np
import pytest

import oracle
from oracle import learned_ref
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def code_of(kind):
    if kind == "one class":
        return inputs.regular_code(40, 20, 3, 6, 5)
    if kind == "many classes":  # column weights 1 .. 18, rows of at most 16 edges
        rng = np.random.default_rng(7)
        sets = [[] for _ in range(60)]
        for j in range(36):
            for i in sorted(range(60), key=lambda i: (len(sets[i]), rng.random()))[:1 + j // 2]:
                sets[i].append(j + 1)
        return inputs.code_from_index_sets([sorted(s) for s in sets], 36)
    base = inputs.irregular_code(40, 20, [2, 3, 4], [0.4, 0.4, 0.2], 21)
    if kind == "short rows":
        return base
    sets = [list(base.cols[base.rows == i] + 1) for i in range(base.M)]
    sets.append(sorted(np.random.default_rng(5).choice(40, 20, replace=False) + 1))
    return inputs.code_from_index_sets(sets, 40)


@pytest.mark.parametrize("frames", [1, 100, 4001, 7900])
@pytest.mark.parametrize("kind", ["short rows", "long row", "one class", "many classes"])
def test_adjoint_over_launch_shapes(kind, frames):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    from paper_2507_10424_gb300.learn import WeightedMinSum
    build.build()
    code = code_of(kind)
    cls, degrees = oracle.column_classes(code)
    assert {"short rows": 3, "long row": 4, "one class": 1, "many classes": 18}[kind] == len(degrees)
    assert (code.row_weights().max() > 16) == (kind == "long row")
    T = 3
    rng = np.random.default_rng(frames)
    a = rng.uniform(0.6, 1.0, (T, len(degrees))).astype(np.float32)
    b = rng.uniform(0.0, 0.3, (T, len(degrees))).astype(np.float32)
    llr = inputs.all_zero_awgn_llr(frames, code.N, 1.5, 0.5, 3)
    w = torch.from_numpy(rng.uniform(0.5, 1.5, (T, frames, code.N)))
    dec = Decoder.from_code(code)
    ta, tb = (torch.from_numpy(x).cuda().requires_grad_() for x in (a, b))
    soft = WeightedMinSum.apply(dec, torch.from_numpy(llr).cuda(), ta, tb, True)
    # twice from the same saved state: the adjoint leaves it as it was
    g1 = torch.autograd.grad(soft, (ta, tb), w.float().cuda(), retain_graph=True)
    g2 = torch.autograd.grad(soft, (ta, tb), w.float().cuda())
    rows = [list(code.cols[code.rows == i]) for i in range(code.M)]
    ra, rb = (torch.from_numpy(x.astype(np.float64)).requires_grad_() for x in (a, b))
    r64 = torch.from_numpy(llr.astype(np.float64))
    ref = torch.stack([learned_ref.unrolled_posteriors(rows, code.N, cls, r64, ra[:t], rb[:t])
                       for t in range(1, T + 1)])
    want = torch.autograd.grad(ref, (ra, rb), w)
    for t in range(T):  # the decode path with the same weights, bit for bit
        dec.set_weights(a, b)
        s = dec.decode(torch.from_numpy(llr).cuda(), t + 1, early_stop=False, want_soft=True)[3]
        assert (s == soft[t]).all()
    for got in (g1, g2):
        for x, y in zip(got, want):
            np.testing.assert_allclose(x.cpu().numpy(), y.numpy(), rtol=0, atol=1e-3 * float(y.abs().max()))
    dec.close()


def test_workspace_of_any_alignment():
    """A caller's workspace on a 4-byte boundary gives the gradients of an aligned one."""
    import torch
    from paper_2507_10424_gb300 import build, ldpc
    from paper_2507_10424_gb300.ldpc import Decoder
    build.build()
    code = inputs.cfg_regular_576()
    dec = Decoder.from_code(code)
    F, T = 2000, 3
    x = torch.from_numpy(inputs.all_zero_awgn_llr(F, code.N, 2.0, 0.5, 3)).cuda()
    a, b = torch.full((T, 1), 0.8, device="cuda"), torch.full((T, 1), 0.1, device="cuda")
    g = torch.randn((F, code.N), device="cuda")
    n = ldpc.ldpc_train_workspace_size(dec.h, F, T)
    work = torch.empty(n + 16, dtype=torch.uint8, device="cuda")
    res = []
    P = lambda t, o=0: ctypes.c_void_p(t.data_ptr() + o)
    for off in (0, 4):
        soft, ga, gb = torch.empty_like(x), torch.empty_like(a), torch.empty_like(b)
        assert ldpc.ldpc_train_forward(dec.h, P(x), F, T, P(a), P(b), P(soft), 0, P(work, off), n) == 0
        assert ldpc.ldpc_train_backward(dec.h, F, T, P(a), P(b), P(g), 0, P(ga), P(gb), P(work, off), n) == 0
        torch.cuda.synchronize()
        res.append((soft, ga, gb))
    assert (res[0][0] == res[1][0]).all()
    for k in (1, 2):
        torch.testing.assert_close(res[0][k], res[1][k], rtol=1e-3, atol=1e-3 * float(res[0][k].abs().max()))
    dec.close()
