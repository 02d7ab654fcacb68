"""The per-path kernels exist with more registers for launches whose blocks all run at once, and with more blocks per SM
for the others (GPU): either side of that line a row, and a node, gets the same bits, and grad_x alone those of the full call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j
from oracle import conv as oconv
from parity_util import assert_blockwise_close, blocks_of_paths

pytestmark = pytest.mark.gpu
SIGNATURES = [("8x0e+8x1o", 2), ("12x0e+12x1o+12x2e", 2), ("8x0e+8x1o+8x2e+8x3o", 3), ("16x0e", 2), ("8x0e+8x0o", 3)]


def _last_small(plan, lmax, real, split):
    """The most rows (nodes) of a forward launch that runs on the kernel with more registers."""
    groups = len({(p["x_off"], p["l2"], lmax == 3 and p["L"] == 3) for p in e3j.e3j_plan_paths(plan)})
    per_sm = 3 if lmax == 3 or real == torch.float64 else 4
    units = plan.n_channels * real.itemsize // 16
    blocks = torch.cuda.get_device_properties(0).multi_processor_count * per_sm // groups
    return blocks * (128 >> split) // units


@pytest.mark.parametrize("irreps,lmax", SIGNATURES)
def test_tensor_products_either_side_of_the_line(irreps, lmax):
    plan = e3j.e3j_plan_create(irreps, lmax, None, lmax)
    assert not plan.specialised
    cp = oconv.Coupling(irreps, lmax, None, lmax)
    rows = _last_small(plan, lmax, torch.float32, 0)
    rng = np.random.default_rng(7)
    host = [rng.standard_normal(s).astype(np.float32) for s in ((rows + 1, plan.d_in, plan.n_channels), (rows + 1, plan.d_sh), (rows + 1, plan.n_paths, plan.n_channels))]
    x, y, w = (torch.from_numpy(a).cuda() for a in host)
    large = e3j.e3j_tp_fwd(plan, x, y, w)
    small = e3j.e3j_tp_fwd(plan, x[:rows], y[:rows], w[:rows])
    assert torch.equal(large[:rows], small)
    ids = np.arange(rows + 1, dtype=np.int32)
    assert_blockwise_close(large.cpu().numpy(), oconv.conv_fwd(cp, *host, ids, ids), blocks_of_paths(cp.paths, "out"), what="out")


@pytest.mark.parametrize("real", [torch.float32, torch.float64])
@pytest.mark.parametrize("irreps,lmax", SIGNATURES)
def test_forwards_either_side_of_the_line(irreps, lmax, real):
    plan = e3j.e3j_plan_create(irreps, lmax, None, lmax)
    cp = oconv.Coupling(irreps, lmax, None, lmax)
    n, degree = _last_small(plan, lmax, real, 3), 6   # (with so few nodes each has eight lanes)
    rng = np.random.default_rng(8)
    rcv = np.repeat(np.arange(n), rng.integers(0, 2 * degree, size=n)).astype(np.int32)
    snd = rng.integers(0, n, size=len(rcv)).astype(np.int32)
    host = [rng.standard_normal(s).astype(np.float32) for s in ((n + 1, plan.d_in, plan.n_channels), (len(rcv), plan.d_sh), (len(rcv), plan.n_paths, plan.n_channels))]
    x, y, w = (torch.from_numpy(a).cuda().to(real) for a in host)
    s, r = torch.from_numpy(snd).cuda(), torch.from_numpy(rcv).cuda()
    call = e3j.e3j_conv_fwd_f64 if real == torch.float64 else e3j.e3j_conv_fwd
    small, large = call(plan, x[:n], y, w, s, r), call(plan, x, y, w, s, r)
    assert torch.equal(large[:n], small) and not large[n].any()
    want = oconv.conv_fwd(cp, host[0][:n], *host[1:], snd, rcv)
    assert_blockwise_close(small.cpu().numpy(), want, blocks_of_paths(cp.paths, "out"), tol=1e-12 if real == torch.float64 else 1e-5, what="out")


@pytest.mark.parametrize("nodes,degree", [(40, 20), (1500, 40)])   # all blocks at once; several waves of them
@pytest.mark.parametrize("real", [torch.float32, torch.float64])
@pytest.mark.parametrize("irreps,lmax", SIGNATURES + [("120x1o", 1)])
def test_grad_x_alone_has_the_bits_of_the_full_call(irreps, lmax, real, nodes, degree):
    plan = e3j.e3j_plan_create(irreps, lmax, None, lmax)
    gen = torch.Generator(device="cuda").manual_seed(9)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=real)
    e = nodes * degree
    r = torch.arange(nodes, device="cuda", dtype=torch.int32).repeat_interleave(degree)
    s = torch.randint(nodes, (e,), generator=gen, device="cuda", dtype=torch.int32)
    _, perm, colptr = e3j.e3j_graph_prepare(nodes, s, r)
    x, sh, w, g = draw(nodes, plan.d_in, plan.n_channels), draw(e, plan.d_sh), draw(e, plan.n_paths, plan.n_channels), draw(nodes, plan.d_out, plan.n_channels)
    lib, f64 = e3j._load(), real == torch.float64
    nbytes = (lib.e3j_conv_f64_workspace_bytes if f64 else lib.e3j_conv_bwd_workspace_bytes)(plan.handle, nodes, e)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

    def call(*wanted):
        grads = [torch.full_like(t, float("nan")) for t in (x, sh, w)]
        ptr = lambda t: t.data_ptr()
        args = [*map(ptr, (x, sh, w, s, r)), *([] if f64 else [None]), *map(ptr, (perm, colptr, g)),
                *(ptr(t) if want else None for t, want in zip(grads, wanted)), ptr(ws), nbytes, torch.cuda.current_stream().cuda_stream]
        assert (lib.e3j_conv_bwd_f64 if f64 else lib.e3j_conv_bwd)(plan.handle, nodes, e, *args) == e3j.E3J_OK
        return grads

    full = call(True, True, True)
    assert not any(t.isnan().any() for t in full)
    for wanted in ((True, False, False), (False, True, False), (False, False, True)):
        assert all(torch.equal(a, b) if want else a.isnan().all() for a, b, want in zip(call(*wanted), full, wanted))
