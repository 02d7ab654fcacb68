"""What the binding allocates, and accepts, as the workspace of a call that may hold the edges' shares of grad_x (no device)."""
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

N, E, HIDDEN = 40, 1000, 8


class _Asked(Exception):
    pass


def _asked_for(monkeypatch, call, *args, **kwargs):
    """The workspace size that a call asks for (tensors on the host: it gets no further)."""
    def workspace(nbytes, *rest):
        raise _Asked(nbytes)
    monkeypatch.setattr(e3j, "_workspace", workspace)
    with pytest.raises(_Asked) as asked:
        call(*args, **kwargs)
    return asked.value.args[0]


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
    assert _asked_for(monkeypatch, e3j.e3j_conv_fwd_f64, plan, x, sh, w, snd, rcv) == graph
    shares = 0 if irreps == "8x0e" else (8 * E * plan.d_in * plan.n_channels + 255) // 256 * 256
    assert e3j.e3j_conv_bwd_shares_bytes(plan, E, 8) == shares
    assert _asked_for(monkeypatch, e3j.e3j_conv_bwd_f64, plan, x, sh, w, snd, rcv, g) == graph + shares
