"""A padded call gives the bits of the plain call whatever the capacity of its list (GPU): how a node's edges are dealt
to runs or lanes must not depend on the number of padding entries."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

pytestmark = pytest.mark.gpu


# 192 nodes of every degree between 0 and twice the mean: senders and receivers on both sides of each threshold of the
# split, lists whose capacity is (1.05, 1.25, 4 times) or is not on the same side of the thresholds as the edge count
@pytest.mark.parametrize("irreps,lmax,specialised", [("128x0e+128x1o", 3, 1), ("32x0e+32x1o", 3, 1), ("12x0e+12x1o+12x2e", 2, 0),
                                                     ("16x0e+16x3o", 3, 0)])
@pytest.mark.parametrize("degree", [7, 20, 47])
def test_padded_results_do_not_depend_on_the_capacity(irreps, lmax, specialised, degree):
    n = 192
    rng = np.random.default_rng(degree)
    plan = e3j.e3j_plan_create(irreps, lmax, None, lmax)
    assert plan.specialised == specialised
    rcv = np.repeat(np.arange(n), rng.permutation(np.arange(n) % (2 * degree + 1))).astype(np.int32)
    e = len(rcv)
    snd = rng.permutation(rcv)
    gen = torch.Generator(device="cuda").manual_seed(degree)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    x, sh, w = draw(n, plan.d_in, plan.n_channels), draw(e, plan.d_sh), draw(e, plan.n_paths, plan.n_channels)
    g = draw(n, plan.d_out, plan.n_channels)
    s, r = torch.from_numpy(snd).cuda(), torch.from_numpy(rcv).cuda()
    rowptr, perm, colptr = e3j.e3j_graph_prepare(n, s, r)
    want = (e3j.e3j_conv_fwd(plan, x, sh, w, s, r, rowptr), *e3j.e3j_conv_bwd(plan, x, sh, w, s, r, g, rowptr, perm, colptr))
    for pad in (0, e // 20, e // 4, 3 * e):
        fill = lambda t, value: torch.cat([t, torch.full((pad, *t.shape[1:]), value, dtype=t.dtype, device="cuda")])
        ps, pr, psh, pw = fill(s, n), fill(r, n), fill(sh, float("nan")), fill(w, float("nan"))
        rowptr, perm, colptr = e3j.e3j_graph_prepare_padded(n, ps, pr)
        got = (e3j.e3j_conv_fwd_padded(plan, x, psh, pw, ps, pr, rowptr),
               *e3j.e3j_conv_bwd_padded(plan, x, psh, pw, ps, pr, g, rowptr, perm, colptr))
        torch.cuda.synchronize()
        for name, a, b in zip(("out", "grad_x", "grad_sh", "grad_w"), got, want):
            assert torch.equal(a[:len(b)], b) and torch.count_nonzero(a[len(b):]) == 0, (name, pad)
