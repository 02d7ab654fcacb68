"""Kernels whose launches overlap the tail of the kernel before them (GPU): calls queued one behind the other, in a
captured graph or without the host ever waiting, give the bits of calls that are waited for one by one; and the binding
gives them with and without its native marshalling."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

pytestmark = pytest.mark.gpu

# per-path kernels (three blocks of inputs; scalars alone), generated ones with staged and with unstaged sender rows
SIGNATURES = [("12x0e+12x1o+12x2e", 2), ("8x0e", 2), ("128x0e+128x1o", 3), ("64x0e+64x1o", 3)]
NODES, EDGES = 120, 1800


class _Case:
    """A list of EDGES edges and everything the calls take, in buffers that new values are copied into."""

    def __init__(self, irreps, lmax):
        self.plan = p = e3j.e3j_plan_create(irreps, lmax, None, lmax)
        self.lmax = lmax
        zeros = lambda *shape: torch.zeros(shape, device="cuda")
        self.ids = [torch.zeros(EDGES, dtype=torch.int32, device="cuda") for _ in range(2)]
        self.x, self.w, self.g = zeros(NODES, p.d_in, p.n_channels), zeros(EDGES, p.n_paths, p.n_channels), zeros(NODES, p.d_out, p.n_channels)
        self.vec = zeros(EDGES, 3)

    def values(self, seed):
        """New ids and arrays (on the host)."""
        rng = np.random.default_rng(seed)
        draw = lambda t: torch.from_numpy(rng.standard_normal(t.shape).astype(np.float32)).pin_memory()
        rcv = np.sort(rng.integers(0, NODES if seed % 2 else NODES // 4, EDGES)).astype(np.int32)
        snd = rng.integers(0, NODES if seed % 3 else 5, EDGES).astype(np.int32)
        return [torch.from_numpy(a).pin_memory() for a in (snd, rcv)] + [draw(t) for t in (self.x, self.w, self.g, self.vec)]

    def load(self, values):
        for dst, src in zip((*self.ids, self.x, self.w, self.g, self.vec), values):
            dst.copy_(src, non_blocking=True)

    def calls(self):
        """One function per call; each takes the results so far and returns its own."""
        plan, (s, r), x, w, g = self.plan, self.ids, self.x, self.w, self.g
        yield "graph", lambda d: e3j.e3j_graph_prepare(NODES, s, r)
        yield "sh", lambda d: (e3j.e3j_harmonics_fwd(self.lmax, self.vec),)
        yield "fwd", lambda d: (e3j.e3j_conv_fwd(plan, x, d["sh"][0], w, s, r, d["graph"][0]),)
        yield "bwd", lambda d: e3j.e3j_conv_bwd(plan, x, d["sh"][0], w, s, r, g, *d["graph"])
        yield "again", lambda d: e3j.e3j_conv_bwd(plan, d["bwd"][0], d["bwd"][1], d["bwd"][2], s, r, d["fwd"][0], *d["graph"])
        yield "vec", lambda d: e3j.e3j_conv_vec_bwd(plan, d["again"][0], self.vec, w, s, r, g, *d["graph"])
        yield "dbl", lambda d: e3j.e3j_conv_bwd_bwd(plan, x, d["sh"][0], w, s, r, g, *d["graph"], *d["bwd"])
        yield "tp", lambda d: e3j.e3j_tp_bwd(plan, x, d["sh"][0][:NODES].contiguous(), w[:NODES].contiguous(), d["dbl"][0])
        if plan.n_channels % 2 == 0:
            f = lambda *a: [t.double() for t in a]
            yield "f64", lambda d: (e3j.e3j_conv_fwd_f64(plan, *f(x, d["sh"][0], w), s, r, d["graph"][0]),
                                    *e3j.e3j_conv_bwd_f64(plan, *f(x, d["sh"][0], w), s, r, *f(g), *d["graph"][1:]))

    def run(self, wait=False):
        done = {}
        for name, call in self.calls():
            done[name] = call(done)
            if wait:
                torch.cuda.synchronize()
        return [t for result in done.values() for t in result]


def _same(got, want):
    assert len(got) == len(want) and all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("irreps,lmax", SIGNATURES)
def test_changing_lists_back_to_back(irreps, lmax):
    case = _Case(irreps, lmax)
    lists = [case.values(seed) for seed in range(8)]
    want = []
    for values in lists:
        case.load(values)
        torch.cuda.synchronize()
        want.append([t.clone() for t in case.run(wait=True)])
    torch.cuda.synchronize()
    got = []
    for values in lists:
        case.load(values)
        got.append(case.run())
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert not any(t.is_floating_point() and t.isnan().any() for t in b)
        _same(a, b)


@pytest.mark.parametrize("irreps,lmax", SIGNATURES)
def test_a_captured_step_follows_its_inputs(irreps, lmax):
    case = _Case(irreps, lmax)
    case.load(case.values(1))
    case.run()   # first use uploads tables and sets the kernels' attributes
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        outputs = case.run()
    for seed in (2, 3, 4):
        case.load(case.values(seed))
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        got = [t.clone() for t in outputs]
        _same(got, case.run(wait=True))


@pytest.mark.parametrize("irreps,lmax", SIGNATURES)
def test_with_and_without_the_native_marshalling(irreps, lmax, monkeypatch):
    case = _Case(irreps, lmax)
    case.load(case.values(5))
    native = case.run()
    assert e3j._native is not None
    monkeypatch.setattr(e3j, "_native", None)
    monkeypatch.setattr(e3j, "_dev_ptr", e3j._dev_ptr_in_python)
    monkeypatch.setattr(e3j, "_empty", e3j._empty_in_python)
    _same(native, case.run())
    parameter = torch.nn.Parameter(case.x)   # not exactly a tensor: the native code hands it to the Python check
    monkeypatch.undo()
    s, r = case.ids
    sh = e3j.e3j_harmonics_fwd(lmax, case.vec)
    with torch.no_grad():
        _same([e3j.e3j_conv_fwd(case.plan, parameter, sh, case.w, s, r)], [e3j.e3j_conv_fwd(case.plan, case.x, sh, case.w, s, r)])
