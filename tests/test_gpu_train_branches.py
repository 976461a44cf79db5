"""GPU tests of the branches of the training kernels that depend on the code's shape: rows of 17
to 27 edges and longer ones (the row and the place of a column's edges in one word or in two
arrays), more rows than edges (a row's gradient pair at its first edges), more than 16 weight
classes with long rows (the class sums by warp reductions), and so many iterations that the
weight gradients' sums take two rounds of the workspace; against autograd in 64 bits.

Tolerance: a gradient entry sums terms that each pass at most T iterations of sums of at most
d + 1 binary32 values, so its error is below 2 T (d + 1) 2^-24 of the sum of the terms'
magnitudes; with T (d + 1) <= 280 and magnitudes summing to at most three times the largest entry
that is 1e-4 of it."""
import numpy as np
import pytest

import oracle
from oracle import learned_ref
from paper_2507_10424_gb300 import inputs

pytestmark = pytest.mark.gpu


def code_of(kind):
    if kind in ("row of 20", "row of 30", "more rows than edges"):
        base = inputs.irregular_code(40, 20, [2, 3, 4], [0.4, 0.4, 0.2], 21)
        sets = [list(base.cols[base.rows == i] + 1) for i in range(base.M)]
        if kind == "more rows than edges":
            return inputs.code_from_index_sets([s for x in sets for s in [[]] * 6 + [x]], 40)
        n = int(kind.split()[-1])
        sets.append(sorted(np.random.default_rng(5).choice(40, n, replace=False) + 1))
        return inputs.code_from_index_sets(sets, 40)
    rng = np.random.default_rng(7)  # column weights 1 .. 18
    sets = [[] for _ in range(60)]
    for j in range(36):
        for i in sorted(range(60), key=lambda i: (len(sets[i]), rng.random()))[:1 + j // 2]:
            sets[i].append(j + 1)
    if kind == "many classes, row of 30":
        sets.append(sorted(rng.choice(36, 30, replace=False) + 1))
    return inputs.code_from_index_sets([sorted(s) for s in sets], 36)


@pytest.mark.parametrize("kind,frames,T", [("row of 20", 70, 3), ("row of 30", 1, 3), ("row of 30", 4001, 3),
                                           ("more rows than edges", 70, 3), ("more rows than edges", 4001, 3),
                                           ("many classes, row of 30", 70, 3), ("many classes", 1, 40)])
def test_gradients(kind, frames, T):
    import torch
    from paper_2507_10424_gb300 import build
    from paper_2507_10424_gb300.ldpc import Decoder
    from paper_2507_10424_gb300.learn import WeightedMinSum
    build.build()
    code = code_of(kind)
    cls, degrees = oracle.column_classes(code)
    E, d = int(code.row_weights().sum()), int(code.row_weights().max())
    if kind == "more rows than edges":
        assert code.M > E
    elif "row of" in kind:
        assert d == int(kind.split()[-1]) and (len(degrees) > 16) == ("many" in kind)
    else:  # fewer iterations' sums than T fit 2 N 32 floats
        assert len(degrees) > 16 and (2 * code.N * 32 * 4 - 8) // (16 * len(degrees)) < T
    rng = np.random.default_rng(frames)
    # (small factors: with up to 18 messages a bit the posteriors would grow without end)
    a = rng.uniform(0.03, 0.05, (T, len(degrees))).astype(np.float32)
    b = rng.uniform(0.0, 0.01, (T, len(degrees))).astype(np.float32)
    llr = inputs.all_zero_awgn_llr(frames, code.N, 1.5, 0.5, 3)
    w = torch.from_numpy(rng.uniform(0.5, 1.5, (frames, code.N)))
    dec = Decoder.from_code(code)
    ta, tb = (torch.from_numpy(x).cuda().requires_grad_() for x in (a, b))
    soft = WeightedMinSum.apply(dec, torch.from_numpy(llr).cuda(), ta, tb, False)
    got = torch.autograd.grad(soft, (ta, tb), w.float().cuda())
    rows = [list(code.cols[code.rows == i]) for i in range(code.M)]
    ra, rb = (torch.from_numpy(x.astype(np.float64)).requires_grad_() for x in (a, b))
    ref = learned_ref.unrolled_posteriors(rows, code.N, cls, torch.from_numpy(llr.astype(np.float64)), ra, rb)
    want = torch.autograd.grad(ref, (ra, rb), w)
    np.testing.assert_allclose(soft.detach().cpu().numpy(), ref.detach().numpy(), rtol=0,
                               atol=1e-4 * float(ref.detach().abs().max()))
    for x, y in zip(got, want):
        np.testing.assert_allclose(x.cpu().numpy(), y.numpy(), rtol=0, atol=1e-4 * float(y.abs().max()))
    dec.close()
