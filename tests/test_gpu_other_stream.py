"""Calls on a stream other than the current one (GPU): what a call allocates for itself is not handed out again before
that stream is done with it, and results that the binding reads are read behind the stream's work."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("irreps,lmax", [("128x0e+128x1o", 3), ("12x0e+12x1o", 2)])
def test_a_workspace_outlives_the_work_on_another_stream(irreps, lmax):
    n, degree = 150, 20
    rng = np.random.default_rng(1)
    plan = e3j.e3j_plan_create(irreps, lmax, None, lmax)
    e = n * degree
    s, r = (torch.from_numpy(a.astype(np.int32)).cuda() for a in (rng.integers(0, n, e), np.repeat(np.arange(n), degree)))
    draw = lambda *shape: torch.randn(shape, device="cuda")
    x, sh, w, g = draw(n, plan.d_in, plan.n_channels), draw(e, plan.d_sh), draw(e, plan.n_paths, plan.n_channels), draw(n, plan.d_out, plan.n_channels)
    want = e3j.e3j_conv_bwd(plan, x, sh, w, s, r, g)     # the sender order is formed in the workspace
    nbytes = e3j.e3j_conv_bwd_workspace_bytes(plan, n, e)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)                    # about 10 ms: the call below waits behind it
    got = e3j.e3j_conv_bwd(plan, x, sh, w, s, r, g, stream=side)
    junk = [torch.zeros(nbytes, dtype=torch.uint8, device="cuda") for _ in range(3)]   # on the current stream, at once
    torch.cuda.synchronize()
    assert len(junk) == 3 and all(torch.equal(a, b) for a, b in zip(got, want))


def test_the_graph_check_reads_its_status_behind_the_stream():
    side = torch.cuda.Stream()
    bad = torch.tensor([3, 1, 2], dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)
    assert e3j.e3j_graph_validate(4, bad, bad, stream=side) == e3j.E3J_ERR_GRAPH
    good = torch.arange(4, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert e3j.e3j_graph_validate(4, good, good, stream=side) == 0


def test_the_shard_count_is_read_behind_the_stream():
    rng = np.random.default_rng(2)
    s = torch.from_numpy(rng.integers(0, 40, 90).astype(np.int32)).cuda()
    r = torch.from_numpy(np.sort(rng.integers(10, 20, 90)).astype(np.int32)).cuda()
    want = e3j.e3j_shard_prepare(40, 10, 20, s, r)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)
    got = e3j.e3j_shard_prepare(40, 10, 20, s, r, stream=side)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
