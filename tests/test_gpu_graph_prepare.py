"""Graph preparation at the edges of its one-launch form (196 608 edges, 262 144 nodes), against numpy (GPU)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

pytestmark = pytest.mark.gpu


# (nodes, edges, padding, nodes that send or receive): one edge; a list without padding and one of padding alone; runs
# of thousands of empty rows before, between and behind; the largest list of the form and the next; a block whose edges
# do not fit; a dense graph; the largest node count of the form and the next; the largest node count whose rows are filled
# from the edges and the next
@pytest.mark.parametrize("n,e,pad,used,hub", [
    (1, 1, 0, 1, 0), (7, 40, 0, 7, 0), (7, 0, 5, 7, 0), (5000, 60, 13, 5000, 0), (70001, 33, 0, 3, 0),
    (3000, 196608, 0, 3000, 0), (3000, 196609, 0, 3000, 0), (100, 20001, 3, 100, 0.5), (100, 100003, 0, 100, 0), (262144, 1000, 7, 262144, 0),
    (262145, 1000, 7, 262145, 0), (65536, 300, 3, 65536, 0), (65537, 300, 3, 65537, 0)])
def test_prepare_matches_numpy(n, e, pad, used, hub):
    rng = np.random.default_rng(n + e)
    ids = np.sort(rng.choice(n, used, replace=False))
    rcv = np.sort(ids[rng.integers(0, used, e)]).astype(np.int32)
    snd = ids[rng.integers(0, used, e)].astype(np.int32)
    if e > 3000:
        snd[: e // 50] = ids[1]    # a hub of some thousand edges
    if hub:
        snd[rng.random(e) < hub] = ids[2]    # more edges than a block collects
    cuda = lambda a, fill: torch.from_numpy(np.concatenate([a, np.full(pad, fill, np.int32)])).cuda()
    prepare = e3j.e3j_graph_prepare_padded if pad else e3j.e3j_graph_prepare
    rowptr, perm, colptr = prepare(n, cuda(snd, n), cuda(rcv, n))
    assert np.array_equal(rowptr.cpu().numpy(), np.searchsorted(rcv, np.arange(n + 1), side="left"))
    assert np.array_equal(perm.cpu().numpy()[:e], np.argsort(snd, kind="stable"))
    assert np.array_equal(colptr.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(snd, minlength=n))]))
    only = prepare(n, cuda(snd, n), cuda(rcv, n), want_transpose=False)
    assert torch.equal(only[0], rowptr) and only[1] is None


def test_a_long_run_of_receivers_without_edges_costs_no_more_than_many_short_ones():
    """The row pointers of 4 million nodes and 1000 edges, spread evenly or all at the two ends: the work is the same
    writes, so the second list may not take several times as long (a run written by one warp took 12 times)."""
    n, e = 4_000_000, 1000
    time = {}
    for kind in ("even", "ends"):
        rcv = np.linspace(0, n - 1, e) if kind == "even" else np.repeat([0, n - 1], e // 2)
        r = torch.from_numpy(rcv.astype(np.int32)).cuda()
        call = lambda: e3j.e3j_graph_prepare(n, r, r, want_transpose=False)
        runs = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                call()
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        time[kind] = min(runs)
    assert time["ends"] < 3 * time["even"], time
