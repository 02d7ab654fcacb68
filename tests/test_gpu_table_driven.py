"""The table-driven kernels against the oracle in every branch they have (GPU): plans that neither generated nor per-path
kernels take, l > 3 or more than 512 channels, through the tensor product, padded lists, collapsed outputs, partial
gradients, the composed double backward and the float64 calls.

Tolerances as in the other parity tests: 1e-5 (float32) and 1e-12 (float64) of an irreducible block's largest value.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j
from oracle import conv as oconv
from parity_util import assert_blockwise_close, blocks_of_paths

pytestmark = pytest.mark.gpu

PLANS = [("8x0e+8x4e", 2, 4), ("516x0e+516x1o", 1, 1)]


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _case(irreps, lmax, out_lmax, flags=0, nodes=9, seed=0):
    rng = np.random.default_rng(seed + len(irreps))
    plan = e3j.e3j_plan_create(irreps, lmax, None, out_lmax, flags)
    cp = oconv.Coupling(irreps, lmax, None, out_lmax)
    rcv = np.repeat(np.arange(nodes), rng.integers(0, 8, nodes)).astype(np.int32)
    snd = rng.integers(0, nodes, len(rcv)).astype(np.int32)
    draw = lambda *shape: rng.standard_normal(shape).astype(np.float32)
    e, c = len(rcv), plan.n_channels
    return plan, cp, snd, rcv, draw(nodes, plan.d_in, c), draw(e, plan.d_sh), draw(e, plan.n_paths, c), draw(nodes, plan.d_out, c)


def _close(cp, got, want, kinds=("out", "x", "sh", "w"), tol=1e-5, blocks={}):
    for have, ref, kind in zip(got, want, kinds):
        assert_blockwise_close(have.cpu().numpy(), ref, blocks.get(kind) or blocks_of_paths(cp.paths, kind), tol=tol, what=kind)


@pytest.mark.parametrize("irreps,lmax,out_lmax", PLANS)
def test_tensor_product(irreps, lmax, out_lmax):
    plan, cp, *_ = _case(irreps, lmax, out_lmax)
    rng, rows, c = np.random.default_rng(3), 37, plan.n_channels
    draw = lambda *shape: rng.standard_normal(shape).astype(np.float32)
    x, y, w, g = draw(rows, plan.d_in, c), draw(rows, plan.d_sh), draw(rows, plan.n_paths, c), draw(rows, plan.d_out, c)
    d = [_cuda(a) for a in (x, y, w, g)]
    want = oconv.tp_bwd(cp, x, y, w, g)
    _close(cp, (e3j.e3j_tp_fwd(plan, *d[:3]), *e3j.e3j_tp_bwd(plan, *d)), (oconv.tp_fwd(cp, x, y, w), *want))
    only_x = e3j.e3j_tp_bwd(plan, *d, grad_x2=False, grad_w=False)
    without_x = e3j.e3j_tp_bwd(plan, *d, grad_x1=False)
    assert only_x[1] is None and only_x[2] is None and without_x[0] is None
    _close(cp, (only_x[0], *without_x[1:]), want, kinds=("x", "sh", "w"))


@pytest.mark.parametrize("irreps,lmax,out_lmax", PLANS)
def test_padded_list_and_partial_gradients(irreps, lmax, out_lmax):
    plan, cp, snd, rcv, x, y, w, g = _case(irreps, lmax, out_lmax)
    n, e, pad = len(x), len(rcv), 13
    dx, dg = _cuda(x), _cuda(g)
    s, r = _cuda(snd), _cuda(rcv)
    rowptr, perm, colptr = e3j.e3j_graph_prepare(n, s, r)
    args = plan, dx, _cuda(y), _cuda(w), s, r
    plain = (e3j.e3j_conv_fwd(*args, rowptr), *e3j.e3j_conv_bwd(*args, dg, rowptr, perm, colptr))
    want = oconv.conv_bwd(cp, x, y, w, snd, rcv, g)
    _close(cp, plain, (oconv.conv_fwd(cp, x, y, w, snd, rcv), *want))
    names = ("grad_x", "grad_sh", "grad_w")
    for kept in names:
        part = e3j.e3j_conv_bwd(*args, dg, rowptr, perm, colptr, **{k: False for k in names if k != kept})
        assert all((t is None) == (k != kept) for t, k in zip(part, names))
        i = names.index(kept)
        assert torch.equal(part[i], plain[1 + i])
    tail = lambda t, value: torch.cat([t, torch.full((pad, *t.shape[1:]), value, dtype=t.dtype, device="cuda")])
    padded = plan, dx, tail(args[2], float("nan")), tail(args[3], float("nan")), tail(s, -5), tail(r, n)
    rowptr, perm, colptr = e3j.e3j_graph_prepare_padded(n, *padded[4:])
    got = (e3j.e3j_conv_fwd_padded(*padded, rowptr), *e3j.e3j_conv_bwd_padded(*padded, dg, rowptr, perm, colptr))
    for a, b in zip(got, plain):
        assert torch.equal(a[:len(b)], b) and torch.count_nonzero(a[len(b):]) == 0


@pytest.mark.parametrize("real", [np.float32, np.float64])
@pytest.mark.parametrize("irreps,lmax,out_lmax", PLANS + [("5x0e+5x1o+5x1e", 2, 2)])
def test_collapsed_outputs(irreps, lmax, out_lmax, real):
    if real is np.float32 and irreps.startswith("5x"):
        pytest.skip("float32 calls take multiples of four channels")
    plan, cp, snd, rcv, x, y, w, g = _case(irreps, lmax, out_lmax, e3j.E3J_PLAN_COLLAPSE_OUTPUTS)
    assert plan.d_out < cp.D
    _, offs = oconv.collapse_matrix(cp)
    blocks = {"out": sorted({(off, off + 2 * p.L + 1) for p, off in zip(cp.paths, offs)})}
    want = (oconv.conv_fwd_collapsed(cp, x, y, w, snd, rcv), *oconv.conv_bwd_collapsed(cp, x, y, w, snd, rcv, g))
    s, r = _cuda(snd), _cuda(rcv)
    rowptr, perm, colptr = e3j.e3j_graph_prepare(len(x), s, r)
    dx, dy, dw, dg = (_cuda(a.astype(real)) for a in (x, y, w, g))
    if real is np.float32:
        got = (e3j.e3j_conv_fwd(plan, dx, dy, dw, s, r, rowptr), *e3j.e3j_conv_bwd(plan, dx, dy, dw, s, r, dg, rowptr, perm, colptr))
    else:
        got = (e3j.e3j_conv_fwd_f64(plan, dx, dy, dw, s, r, rowptr), *e3j.e3j_conv_bwd_f64(plan, dx, dy, dw, s, r, dg, perm, colptr))
    _close(cp, got, want, tol=1e-5 if real is np.float32 else 1e-12, blocks=blocks)


@pytest.mark.parametrize("irreps,lmax,out_lmax", PLANS)
def test_composed_double_backward(irreps, lmax, out_lmax):
    plan, cp, snd, rcv, x, y, w, g = _case(irreps, lmax, out_lmax)
    rng = np.random.default_rng(11)
    cts = [rng.standard_normal(a.shape).astype(np.float32) for a in (x, y, w)]
    s, r = _cuda(snd), _cuda(rcv)
    prep = e3j.e3j_graph_prepare(len(x), s, r)
    got = e3j.e3j_conv_bwd_bwd(plan, _cuda(x), _cuda(y), _cuda(w), s, r, _cuda(g), *prep, *map(_cuda, cts))
    _close(cp, got, oconv.conv_bwd_bwd(cp, x, y, w, snd, rcv, g, *cts))
