"""The per-path kernels (plans without generated ones) against the oracle, at the edges of their ranges (GPU).

Tolerances as in the other parity tests: 1e-5 (float32) and 1e-12 (float64) of an irreducible block's largest value.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j
from oracle import conv as oconv
from parity_util import assert_blockwise_close, blocks_of_paths

pytestmark = pytest.mark.gpu

# (irreps, lmax, out_lmax, float64 only, nodes, mean degree): one unit of four channels; 11 units with every l up to 3
# and two irreps of one l; an irrep no path reads; 128 units, the most a block takes, and one more (table-driven);
# l = 4 (table-driven); a channel count that is odd; enough nodes that a node's edges are not dealt to several lanes
CASES = [("4x0e", 1, 1, 0, 5, 3), ("44x0e+44x1o+44x1e+44x2e+44x3o", 3, 3, 0, 40, 9),
         ("12x0e+12x1o+12x2e+12x3o", 1, 1, 0, 33, 20), ("512x1o", 1, 1, 0, 7, 6), ("516x0e", 1, 1, 0, 7, 6),
         ("8x4e", 1, 4, 0, 20, 8), ("5x1o", 2, 2, 1, 20, 8), ("20x0e+20x1o", 2, 2, 0, 3001, 2)]


@pytest.mark.parametrize("real", [np.float32, np.float64])
@pytest.mark.parametrize("irreps,lmax,out_lmax,f64_only,nodes,degree", CASES)
def test_against_the_oracle(irreps, lmax, out_lmax, f64_only, nodes, degree, real):
    if f64_only and real is np.float32:
        pytest.skip("float32 calls take multiples of four channels")
    rng = np.random.default_rng(len(irreps) + nodes)
    plan = e3j.e3j_plan_create(irreps, lmax, None, out_lmax)
    assert not plan.specialised
    cp = oconv.Coupling(irreps, lmax, None, out_lmax)
    degrees = rng.integers(0, 2 * degree + 1, size=nodes)   # nodes without edges among them
    rcv = np.repeat(np.arange(nodes), degrees).astype(np.int32)
    e = len(rcv)
    snd = rng.integers(0, nodes, size=e).astype(np.int32)
    draw = lambda *shape: rng.standard_normal(shape).astype(np.float32)
    x, y, w, g = (draw(nodes, plan.d_in, plan.n_channels), draw(e, plan.d_sh), draw(e, plan.n_paths, plan.n_channels),
                  draw(nodes, plan.d_out, plan.n_channels))
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    s, r = cuda(snd), cuda(rcv)
    graph = e3j.e3j_graph_prepare(nodes, s, r)
    if real is np.float32:
        d = [cuda(a) for a in (x, y, w, g)]
        call = lambda: (e3j.e3j_conv_fwd(plan, *d[:3], s, r, graph[0]), *e3j.e3j_conv_bwd(plan, *d[:3], s, r, d[3], *graph))
        tol = 1e-5
    else:
        # arrays at the start of their storage, then 8 bytes into it: the second call cannot use 16-byte loads
        def place(a, off):
            t = torch.empty(a.size + 2, dtype=torch.float64, device="cuda")[off:off + a.size].view(a.shape)
            t.copy_(torch.from_numpy(a))
            return t
        d = [place(a, 0) for a in (x, y, w, g)]
        m = [place(a, 1) for a in (x, y, w, g)]
        both = lambda v: (e3j.e3j_conv_fwd_f64(plan, *v[:3], s, r, graph[0]),
                          *e3j.e3j_conv_bwd_f64(plan, *v[:3], s, r, v[3], *graph[1:]))
        call, tol = (lambda: both(d)), 1e-12
    got, again = call(), call()
    want = (oconv.conv_fwd(cp, x, y, w, snd, rcv), *oconv.conv_bwd(cp, x, y, w, snd, rcv, g))
    results = [got] if real is np.float32 else [got, both(m)]
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, again))
    for res in results:
        for have, ref, kind in zip(res, want, ("out", "x", "sh", "w")):
            assert_blockwise_close(have.cpu().numpy(), ref, blocks_of_paths(cp.paths, kind), tol=tol, what=kind)
    unread = np.ones(plan.d_in, bool)
    for lo, hi in blocks_of_paths(cp.paths, "x"):
        unread[lo:hi] = False
    assert all((res[1][:, torch.from_numpy(unread).cuda()] == 0).all() for res in results)


@pytest.mark.parametrize("rows", [1, 257])
def test_tensor_product_rows(rows):
    plan = e3j.e3j_plan_create("12x0e+12x1o+12x3o", 3, None, 3)
    assert not plan.specialised
    gen = torch.Generator(device="cuda").manual_seed(rows)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    x, y, w = draw(rows, plan.d_in, 12), draw(rows, plan.d_sh), draw(rows, plan.n_paths, 12)
    g = draw(rows, plan.d_out, 12)
    ids = torch.arange(rows, dtype=torch.int32, device="cuda")
    graph = e3j.e3j_graph_prepare(rows, ids, ids)
    same = lambda a, b: torch.testing.assert_close(a, b, rtol=1e-5, atol=1e-5)
    same(e3j.e3j_tp_fwd(plan, x, y, w), e3j.e3j_conv_fwd(plan, x, y, w, ids, ids, graph[0]))
    for a, b in zip(e3j.e3j_tp_bwd(plan, x, y, w, g), e3j.e3j_conv_bwd(plan, x, y, w, ids, ids, g, *graph)):
        same(a, b)
