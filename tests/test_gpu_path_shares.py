"""The backward of plans without generated kernels with and without room for the edges' shares of grad_x, and the forward
by pairs under output filters, against the oracle (GPU).  Tolerances as in the other parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j
from oracle import conv as oconv
from parity_util import assert_blockwise_close, blocks_of_paths

pytestmark = pytest.mark.gpu


def _case(irreps, lmax, out, nodes, degree, real):
    rng = np.random.default_rng(nodes + degree)
    plan = e3j.e3j_plan_create(irreps, lmax, out, -1 if out else lmax)
    assert not plan.specialised
    cp = oconv.Coupling(irreps, lmax, out, None if out else lmax)
    rcv = np.repeat(np.arange(nodes), rng.integers(0, 2 * degree + 1, size=nodes)).astype(np.int32)   # some without edges
    snd = rng.integers(0, nodes, size=len(rcv)).astype(np.int32)
    draw = lambda *shape: rng.standard_normal(shape).astype(np.float32)
    host = (draw(nodes, plan.d_in, plan.n_channels), draw(len(rcv), plan.d_sh), draw(len(rcv), plan.n_paths, plan.n_channels),
            draw(nodes, plan.d_out, plan.n_channels))
    dev = [torch.from_numpy(a).cuda().to(real) for a in host]
    return plan, cp, snd, rcv, host, dev


# one unit; 11 units of a node's row to a warp and every l; an irrep no path reads; 128 units; enough nodes for one lane
# each; a hub (few nodes, many edges each)
@pytest.mark.parametrize("real", [torch.float32, torch.float64])
@pytest.mark.parametrize("irreps,lmax,nodes,degree", [("4x1o", 1, 1, 2), ("44x0e+44x1o+44x2e+44x3o", 3, 33, 9), ("12x0e+12x1o+12x3o", 1, 40, 20),
                                                      ("256x0e+256x1o", 2, 5, 7), ("8x0e+8x1o", 2, 3001, 2), ("8x1o+8x2e", 3, 2, 300)])
def test_with_and_without_room_for_the_shares(irreps, lmax, nodes, degree, real):
    plan, cp, snd, rcv, host, (x, sh, w, g) = _case(irreps, lmax, None, nodes, degree, real)
    e, size = len(rcv), x.element_size()
    s, r = torch.from_numpy(snd).cuda(), torch.from_numpy(rcv).cuda()
    rowptr, perm, colptr = e3j.e3j_graph_prepare(nodes, s, r)
    lib, f64 = e3j._load(), real == torch.float64
    query = lib.e3j_conv_f64_workspace_bytes if f64 else lib.e3j_conv_bwd_workspace_bytes
    full = query(plan.handle, nodes, e)
    least = full - (size * e * plan.d_in * plan.n_channels + 255) // 256 * 256

    def call(nbytes, want_x=True):
        grads = [torch.full_like(t, float("nan")) for t in (x, sh, w)]
        ws = torch.full((max(nbytes, 256),), 255, dtype=torch.uint8, device="cuda")
        p = [t.data_ptr() for t in (x, sh, w, s, r, rowptr, perm, colptr, g, *grads, ws)]
        if not want_x:
            p[9] = None
        if f64:
            del p[5]
        status = (lib.e3j_conv_bwd_f64 if f64 else lib.e3j_conv_bwd)(plan.handle, nodes, e, *p, nbytes,
                                                                     torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return status, grads

    want = oconv.conv_bwd(cp, *host[:3], snd, rcv, host[3])
    (s0, shares), (s1, again), (s2, inputs) = call(full), call(full), call(least)
    assert (s0, s1, s2) == (e3j.E3J_OK,) * 3
    assert all(torch.equal(a, b) for a, b in zip(shares, again))
    assert all(torch.equal(a, b) for a, b in zip(shares[1:], inputs[1:]))
    for res in (shares, inputs):
        for have, ref, kind in zip(res, want, ("x", "sh", "w")):
            assert_blockwise_close(have.cpu().numpy(), ref, blocks_of_paths(cp.paths, kind), tol=1e-12 if f64 else 1e-5, what=kind)
    _, edges = call(full, want_x=False)
    assert edges[0].isnan().all() and all(torch.equal(a, b) for a, b in zip(shares[1:], edges[1:]))
    if not f64:
        assert call(least - 256)[0] == e3j.E3J_ERR_WORKSPACE


# filters that leave a pair its lowest, middle or highest output only, or none
@pytest.mark.parametrize("out", ["0e+1o+2e+3o", "1o", "3o+3e", "2e+0e", "2o+1e"])
@pytest.mark.parametrize("irreps,lmax", [("12x0e+12x1o+12x2e+12x3o", 3), ("20x1o+20x1e+20x2e", 2)])
def test_output_filters(irreps, lmax, out):
    plan, cp, snd, rcv, host, (x, sh, w, g) = _case(irreps, lmax, out, 50, 11, torch.float32)
    s, r = torch.from_numpy(snd).cuda(), torch.from_numpy(rcv).cuda()
    graph = e3j.e3j_graph_prepare(50, s, r)
    got = (e3j.e3j_conv_fwd(plan, x, sh, w, s, r, graph[0]), *e3j.e3j_conv_bwd(plan, x, sh, w, s, r, g, *graph))
    want = (oconv.conv_fwd(cp, *host[:3], snd, rcv), *oconv.conv_bwd(cp, *host[:3], snd, rcv, host[3]))
    for have, ref, kind in zip(got, want, ("out", "x", "sh", "w")):
        assert_blockwise_close(have.cpu().numpy(), ref, blocks_of_paths(cp.paths, kind), what=kind)


def test_calls_with_a_backward_run_on_a_workspace_without_the_room():
    """Through the binding: the same edge gradients to the bit, the same grad_x up to the order of its sums."""
    plan, cp, snd, rcv, host, (x, sh, w, g) = _case("12x0e+12x1o+12x2e", 2, None, 40, 12, torch.float32)
    n, e, hidden = 40, len(rcv), 8
    s, r = torch.from_numpy(snd).cuda(), torch.from_numpy(rcv).cuda()
    graph = e3j.e3j_graph_prepare(n, s, r)
    gen = torch.Generator(device="cuda").manual_seed(1)
    vec = torch.randn(e, 3, generator=gen, device="cuda")
    h, W = torch.randn(e, hidden, generator=gen, device="cuda"), torch.randn(hidden, plan.n_paths * plan.n_channels, generator=gen, device="cuda")
    calls = [
        (e3j.e3j_conv_bwd_workspace_bytes(plan, n, e), lambda **k: e3j.e3j_conv_bwd(plan, x, sh, w, s, r, g, *graph, **k)),
        (e3j.e3j_conv_bwd_workspace_bytes(plan, n, e), lambda **k: e3j.e3j_conv_bwd_padded(plan, x, sh, w, s, r, g, *graph, **k)),
        (e3j.e3j_conv_vec_bwd_workspace_bytes(plan, n, e), lambda **k: e3j.e3j_conv_vec_bwd(plan, x, vec, w, s, r, g, *graph, **k)),
        (e3j.e3j_conv_radial_bwd_workspace_bytes(plan, n, e, hidden), lambda **k: e3j.e3j_conv_radial_bwd(plan, x, sh, h, W, s, r, g, *graph, **k)),
        (e3j.e3j_conv_radial_vec_bwd_workspace_bytes(plan, n, e, hidden), lambda **k: e3j.e3j_conv_radial_vec_bwd(plan, x, vec, h, W, s, r, g, *graph, **k)),
        (e3j.e3j_conv_bwd_bwd_workspace_bytes(plan, n, e), lambda **k: tuple(e3j.e3j_conv_bwd_bwd(plan, x, sh, w, s, r, g, *graph, x, sh, w, **k)[i] for i in (1, 0, 2, 3))),
    ]
    room = e3j.e3j_conv_bwd_shares_bytes(plan, e)
    assert room >= 4 * e * plan.d_in * plan.n_channels
    for nbytes, call in calls:
        full = call()
        for size in (nbytes, nbytes - room):
            ws = torch.full((size,), 255, dtype=torch.uint8, device="cuda")
            grads = call(workspace=ws)
            assert all(torch.equal(a, b) for a, b in zip(grads[1:], full[1:]))
            assert torch.equal(grads[0], full[0]) or size < nbytes
            assert_blockwise_close(grads[0].cpu().numpy(), full[0].cpu().numpy(), blocks_of_paths(cp.paths, "x"), what="x")
        with pytest.raises(ValueError):
            call(workspace=ws[:nbytes - room - 256])
