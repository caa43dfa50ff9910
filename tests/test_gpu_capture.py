"""A scan's own calls captured in a CUDA graph by the program: the kernels counted are
those of the graph, and replays of it give the oracle's counts and hulls.  Thin
paths on whole planes and strips, thick rays by both readings and on the plans the
tiled path does not take, one method alone, and page-locked inputs (read in place
while capturing)."""
import ctypes

import numpy as np
import pytest

from paper_1402_1720_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

G = synth.Geometry
VP = ctypes.c_void_p


@pytest.fixture(scope="module")
def hd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1402_1720_gb300 import hulld
    hulld.load()
    return hulld


class _Graph:
    """What a stream is given while it captures, through the driver."""

    def __init__(self, stream):
        self.cu, self.stream = ctypes.CDLL("libcuda.so.1"), VP(stream.cuda_stream)

    def _ok(self, r):
        assert r == 0, r

    def __enter__(self):
        self._ok(self.cu.cuStreamBeginCapture_v2(self.stream, 1))  # thread local
        return self

    def __exit__(self, *exc):
        self.graph = VP()
        r = self.cu.cuStreamEndCapture(self.stream, ctypes.byref(self.graph))
        if exc[0] is None:
            self._ok(r)

    def kernels(self):
        n = ctypes.c_size_t()
        self._ok(self.cu.cuGraphGetNodes(self.graph, None, ctypes.byref(n)))
        nodes = (VP * n.value)()
        self._ok(self.cu.cuGraphGetNodes(self.graph, nodes, ctypes.byref(n)))
        kinds = []
        for node in nodes:
            t = ctypes.c_int()
            self._ok(self.cu.cuGraphNodeGetType(VP(node), ctypes.byref(t)))
            kinds.append(t.value)
        return kinds.count(0)

    def run(self, times):
        ex = VP()
        self._ok(self.cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), self.graph, ctypes.c_ulonglong(0)))
        for _ in range(times):
            self._ok(self.cu.cuGraphLaunch(ex, self.stream))
        torch.cuda.synchronize()
        self._ok(self.cu.cuGraphExecDestroy(ex))
        self._ok(self.cu.cuGraphDestroy(self.graph))


CASES = [
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 7, "thin", None),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 4, "thin", None),
    (G(300, 250, 50, 0.2, 0.2, 0.5, 60.0), 7, "thin", None),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 7, "thick", None),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 2, "thick", None),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 7, "thick", (512, 12, 32767, 3)),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 7, "distance", None),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 4, "distance", None),
    (G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), 7, "distance", (512, 12, 32767, 3)),
]


@pytest.mark.parametrize("g,methods,how,tuning", CASES)
@pytest.mark.parametrize("pinned", [False, True])
def test_captured_scan(hd, oracle_mod, g, methods, how, tuning, pinned):
    n = 5000
    h = synth.tiny_random_case(np.random.default_rng(g.nx), n, g, span=1.1)
    ref = {"thin": lambda: oracle_mod.run(g, h), "thick": lambda: oracle_mod.run_thick(g, h, 2),
           "distance": lambda: oracle_mod.run_euclid(g, h, 1.3, threads=16)}[how]()
    cols = [torch.from_numpy(np.ascontiguousarray(a)) for a in h.arrays()]
    cols = [c.pin_memory() if pinned else c.cuda() for c in cols]
    p = hd.hd_params_default()
    p.methods = methods
    V, st = g.nx * g.ny * g.nz, torch.cuda.Stream()
    mask = torch.zeros(V, dtype=torch.uint8, device="cuda")
    counts = torch.zeros(V, dtype=torch.int32, device="cuda")
    which = hd.HD_SM if methods & 4 else hd.HD_MSC
    with hd.Scan(g, p) as s:
        if tuning is not None:
            hd.hd_scan_set_tuning(s.handle, hd.hd_tuning(*tuning))
        if how == "thick":
            s.set_thick(2)
        if how == "distance":
            s.set_thick_distance(1.3)

        def calls():
            s.reset(st)
            s.add(cols, st)
            s.finalize(st)
            s.mask(which, out=mask, stream=st)
            s.counts(which, out=counts, stream=st)
        torch.cuda.synchronize()
        calls()  # buffers and descriptor
        torch.cuda.synchronize()
        mask.zero_(), counts.zero_()
        torch.cuda.synchronize()
        before = s.profile()["kernel_launches"]
        with _Graph(st) as graph:
            calls()
        assert s.profile()["kernel_launches"] - before == graph.kernels()
        graph.run(2)
        assert np.array_equal(mask.cpu().numpy(), ref["H3" if methods & 4 else "H2"])
        assert np.array_equal(counts.cpu().numpy().view(np.uint32), ref["M" if methods & 4 else "N"])


def test_captured_batch(hd, oracle_mod):
    """A batch's own count, of the kernels another capture of the same run takes."""
    grids = [G(40, 36, 9, 1.0, 1.0, 2.0, 40.0), G(64, 20, 30, 1.0, 1.0, 1.0, 50.0)]
    hs = [synth.tiny_random_case(np.random.default_rng(k), 3000, g, span=1.1) for k, g in enumerate(grids)]
    devs = [[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in h.arrays()] for h in hs]
    st, scans = torch.cuda.Stream(), [hd.Scan(g) for g in grids]
    torch.cuda.synchronize()
    flags = hd.HD_BATCH_RESET | hd.HD_BATCH_FINALIZE
    with hd.Batch() as b:
        counted = []
        for graph in (True, True, False):
            b.set_graph(graph)
            for s, d in zip(scans, devs):
                b.add(s, d)
            before = b.stats()["kernel_launches"]
            b.run(flags, st)
            torch.cuda.synchronize()
            counted.append(b.stats()["kernel_launches"] - before)
    # per scan reset, begin, ingest, scatter and two of the decisions; one traversal, one global pass
    assert counted == [14, 14, 14]
    for s, g, h in zip(scans, grids, hs):
        assert np.array_equal(s.counts(hd.HD_MSC), oracle_mod.run(g, h)["N"])
        s.close()


def test_captured_page_locked_add_of_many(hd):
    """As many page-locked histories as are copied beside the traversal: read in place when
    the stream is capturing."""
    n, g = (3 << 20) + 5, G(24, 20, 12, 1.0, 1.0, 2.0, 30.0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    u = torch.rand((6, n), generator=gen, device="cuda")
    u[0] *= 360.0
    u[1:5] = 24.0 * u[1:5] - 12.0
    u[5] *= 10.0
    host = torch.empty((6, n), pin_memory=True).copy_(u)
    st = torch.cuda.Stream()
    out = [torch.zeros(24 * 20 * 12, dtype=torch.int32, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    with hd.Scan(g) as s:
        s.add([u[k] for k in range(6)])
        s.counts(hd.HD_MSC, out=out[0])
        torch.cuda.synchronize()
        before = s.profile()["kernel_launches"]
        with _Graph(st) as graph:
            s.reset(st)
            s.add([host[k] for k in range(6)], st)
            s.counts(hd.HD_MSC, out=out[1], stream=st)
        assert s.profile()["kernel_launches"] - before == graph.kernels() == 7
        graph.run(2)
    assert torch.equal(*out) and int(out[0].sum()) > 0
