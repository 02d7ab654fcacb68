"""What the binding allocates, and accepts, as the workspace of a call that may hold the edges' shares of grad_x (no device)."""
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

N, E, HIDDEN = 40, 1000, 8


class _Asked(Exception):
    pass


def _asked_for(monkeypatch, call, *args, **kwargs):
    """The workspace size that a call asks for, and the smallest it takes from its caller (tensors on the host: it gets no
    further)."""
    def workspace(nbytes, like, given, stream, least=None):
        raise _Asked(nbytes, least() if least else nbytes)
    monkeypatch.setattr(e3j, "_workspace", workspace)
    with pytest.raises(_Asked) as asked:
        call(*args, **kwargs)
    return asked.value.args


def _inputs(plan, real=torch.float32):
    ids = torch.zeros(E, dtype=torch.int32)
    return (torch.zeros(N, plan.d_in, plan.n_channels, dtype=real), torch.zeros(E, plan.d_sh, dtype=real),
            torch.zeros(E, plan.n_paths, plan.n_channels, dtype=real), ids, ids,
            torch.zeros(N, plan.d_out, plan.n_channels, dtype=real))


@pytest.mark.parametrize("irreps", ["48x0e+48x1o+48x2e", "128x0e+128x1o", "8x0e"])
def test_the_float64_forward_takes_the_graph_arrays_only(irreps, monkeypatch):
    plan = e3j.e3j_plan_create(irreps, 2, None, 2)
    x, sh, w, snd, rcv, g = _inputs(plan, torch.float64)
    graph = 2 * ((4 * (N + 1) + 255) // 256 * 256) + (4 * E + 255) // 256 * 256
    assert _asked_for(monkeypatch, e3j.e3j_conv_fwd_f64, plan, x, sh, w, snd, rcv)[0] == graph
    shares = 0 if irreps == "8x0e" else (8 * E * plan.d_in * plan.n_channels + 255) // 256 * 256
    assert e3j.e3j_conv_bwd_shares_bytes(plan, E, 8) == shares
    assert _asked_for(monkeypatch, e3j.e3j_conv_bwd_f64, plan, x, sh, w, snd, rcv, g)[0] == graph + shares


def _backwards(plan):
    """(call, its workspace query) of everything that contains a backward."""
    x, sh, w, snd, rcv, g = _inputs(plan)
    vec, h = torch.zeros(E, 3), torch.zeros(E, HIDDEN)
    W = torch.zeros(HIDDEN, plan.n_paths * plan.n_channels)
    return {
        "conv": (lambda **k: e3j.e3j_conv_bwd(plan, x, sh, w, snd, rcv, g, **k), e3j.e3j_conv_bwd_workspace_bytes(plan, N, E)),
        "padded": (lambda **k: e3j.e3j_conv_bwd_padded(plan, x, sh, w, snd, rcv, g, snd, snd, snd, **k), e3j.e3j_conv_bwd_workspace_bytes(plan, N, E)),
        "vec": (lambda **k: e3j.e3j_conv_vec_bwd(plan, x, vec, w, snd, rcv, g, **k), e3j.e3j_conv_vec_bwd_workspace_bytes(plan, N, E)),
        "radial": (lambda **k: e3j.e3j_conv_radial_bwd(plan, x, sh, h, W, snd, rcv, g, **k),
                   e3j.e3j_conv_radial_bwd_workspace_bytes(plan, N, E, HIDDEN)),
        "radial_vec": (lambda **k: e3j.e3j_conv_radial_vec_bwd(plan, x, vec, h, W, snd, rcv, g, **k),
                       e3j.e3j_conv_radial_vec_bwd_workspace_bytes(plan, N, E, HIDDEN)),
    }


@pytest.mark.parametrize("call", ["conv", "padded", "vec", "radial", "radial_vec"])
@pytest.mark.parametrize("irreps", ["48x0e+48x1o+48x2e", "128x0e+128x1o"])
def test_no_room_for_shares_of_a_gradient_that_is_not_wanted(irreps, call, monkeypatch):
    plan = e3j.e3j_plan_create(irreps, 2, None, 2)
    shares = e3j.e3j_conv_bwd_shares_bytes(plan, E)
    assert (shares > 0) == (not plan.specialised)
    run, full = _backwards(plan)[call]
    assert _asked_for(monkeypatch, run)[0] == full
    assert _asked_for(monkeypatch, run, workspace=torch.empty(1)) == (full, full - shares)
    assert _asked_for(monkeypatch, run, grad_x=False) == (full - shares, full - shares)


def test_the_double_backward_takes_a_workspace_without_the_room(monkeypatch):
    plan = e3j.e3j_plan_create("48x0e+48x1o+48x2e", 2, None, 2)
    x, sh, w, snd, rcv, g = _inputs(plan)
    full = e3j.e3j_conv_bwd_bwd_workspace_bytes(plan, N, E)
    asked = _asked_for(monkeypatch, e3j.e3j_conv_bwd_bwd, plan, x, sh, w, snd, rcv, g, None, None, None, x, sh, w, workspace=torch.empty(1))
    assert asked == (full, full - e3j.e3j_conv_bwd_shares_bytes(plan, E)) and asked[1] < asked[0]


@pytest.mark.parametrize("element", [4, 8])
def test_the_room_ends_at_two_gib(element):
    plan = e3j.e3j_plan_create("120x0e+120x1o+120x2e+120x3o", 3, None, 3)
    row = element * plan.d_in * plan.n_channels
    longest = (2 << 30) // row
    query = e3j._load().e3j_conv_f64_workspace_bytes if element == 8 else e3j._load().e3j_conv_bwd_workspace_bytes
    full = lambda edges: query(plan.handle, N, edges)
    room = lambda edges: e3j.e3j_conv_bwd_shares_bytes(plan, edges, element)
    assert longest * row <= room(longest) <= 2 << 30 and room(longest + 1) == 0
    assert full(longest + 1) < 24 * longest < full(longest)
    # what the call needs grows with the list all the same: a workspace for a long one serves every shorter one
    needs = [full(edges) - room(edges) for edges in (0, 1, longest - 1, longest, longest + 1, 5_000_000)]
    assert needs == sorted(needs)
    assert room(0) == 0 and e3j.e3j_conv_bwd_shares_bytes(plan, 10, 2) == 0
