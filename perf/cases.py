"""The work a user of this library has it do, as cases that can be timed.

A case is one pass through the public binding (paper_1402_1720_gb300.hulld):
a scan from its histories to its hulls (thin paths, thick rays, one call or
per-angle chunks, device or page-locked host inputs), several scans in one
batch, served scans, the rows of the hull-restricted system matrix, the binned
variant of space carving, and the hull diagnostics.  Inputs are proton
histories of ellipsoid phantoms made on the GPU from a seed: uniform entry
positions on the tracker face, Gaussian exit displacement, WEPL the RSP line
integral plus noise, grouped by gantry angle as an acquisition delivers them.

Every output is a whole number (counts, hull bytes, voxel indices, bin sums).
"""
import math

import numpy as np
import torch

from paper_1402_1720_gb300 import hulld as H
from paper_1402_1720_gb300 import synth

METHODS = (H.HD_SC, H.HD_MSC, H.HD_SM)


def _case(name, kind, grid, voxel, T, angles, per_angle, phantom="head", u_half=0.0, v_half=0.0,
          sigma=2.0, methods=7, chunks=1, pinned=False, thick=0, d0=0.0, scans=1):
    """u_half, v_half: half the tracker face (mm); 0 covers the volume's in-plane diagonal and
    its height.  chunks: add calls the histories arrive in.  thick: in-plane dilation in
    voxels.  d0: Euclidean thickness in mm.  scans: scans of a batch or a serving pass."""
    nx, ny, nz = grid
    sx, sy, sz = voxel
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "sx": sx, "sy": sy,
            "sz": sz, "T": T, "angles": angles, "per_angle": per_angle, "phantom": phantom,
            "u_half": u_half, "v_half": v_half, "sigma": sigma, "methods": methods,
            "chunks": chunks, "pinned": pinned, "thick": thick, "d0": d0, "scans": scans}


def listed():
    head = dict(grid=(200, 200, 32), voxel=(1.0, 1.0, 2.5), T=155.0, u_half=141.5, v_half=40.0)
    return [
        # a quick look at a small object, all three methods: launches and latency count
        _case("tiny", "scan", (64, 64, 8), (1.0, 1.0, 2.5), 100.0, 90, 2000, "ellipsoid", 35.0,
              10.0, 1.0),
        # the ordinary scan: a head-sized volume, the whole acquisition in one call
        _case("head", "scan", angles=90, per_angle=100_000, **head),
        # the same scan read from page-locked host memory, hulls returned to the host
        _case("head_host", "scan", angles=90, per_angle=100_000, pinned=True, **head),
        # a ragged grid and one method alone (MSC), as a preprocessing step asks for it
        _case("ragged_msc", "scan", (181, 217, 37), (0.93, 0.93, 1.9), 150.0, 75, 40_013,
              methods=H.HD_MSC),
        # a large volume streamed per gantry angle while the acquisition runs
        _case("streamed", "scan", (400, 400, 128), (0.5, 0.5, 1.25), 155.0, 60, 550_000,
              u_half=141.5, v_half=80.0, chunks=60),
        # many uneven scans in one batched launch (three grids, random phantoms)
        _case("batch", "batch", (128, 128, 32), (1.0, 1.0, 2.5), 101.0, 90, 10_000, "random",
              scans=12),
        # scans served from per-angle host chunks as they arrive
        _case("served", "served", (128, 128, 32), (1.0, 1.0, 2.5), 101.0, 90, 6_000, "random",
              scans=4),
        # the system-matrix rows an iterative solver reads, inside the MSC hull
        _case("rows", "rows", angles=90, per_angle=20_000, methods=H.HD_MSC, **head),
        # space carving with bins and data cuts on the whole head-sized acquisition
        _case("binned", "binned", angles=90, per_angle=100_000, **head),
        # thick rays dilated in-plane
        _case("thick", "scan", angles=90, per_angle=100_000, thick=2, **head),
        # thick rays by Euclidean distance, reaching across slices
        _case("euclid", "scan", angles=90, per_angle=30_000, d0=2.5, **head),
        # what follows a scan: enclosed hull, edge threshold, comparison, voxel list
        _case("diagnostics", "diagnostics", angles=90, per_angle=20_000, **head),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan"] * 4 + ["chunks", "host", "batch", "served", "rows", "rows",
                                      "binned", "thick", "thick", "euclid", "euclid", "euclid",
                                      "diagnostics"])
    large = kind in ("scan", "chunks") and rng.random() < 0.3
    nx, ny = (_log_int(rng, 257, 400) if large else _log_int(rng, 48, 256) for _ in range(2))
    nz = _log_int(rng, 6, 128) if large else _log_int(rng, 6, 64)
    s = max(0.5, rng.uniform(60.0, 200.0) / max(nx, ny))
    sz = rng.choice([1.0, 1.25, 2.5, rng.uniform(0.8, 3.0)])
    angles = rng.choice([45, 60, 72, 90, 180])
    most = {"scan": 9e6, "chunks": 9e6, "host": 9e6, "batch": 6e5, "served": 4e5, "rows": 1.8e6,
            "binned": 9e6, "thick": 6e6, "euclid": 1e6, "diagnostics": 1e6}[kind]
    per = max(1, _log_int(rng, 2e5, most) // angles)
    phantom = rng.choice(["head", "ellipsoid", "random"])
    T = math.ceil(math.hypot(nx * s, ny * s) / 2 + 10.0)
    methods = 7 if rng.random() < 0.7 else rng.choice([1, 2, 4, 3, 6])
    case = _case("", "scan" if kind in ("chunks", "host", "thick", "euclid") else kind,
                 (nx, ny, nz), (s, s, sz), float(T), angles, per, phantom,
                 sigma=rng.choice([1.0, 2.0, 3.0]),
                 methods=7 if kind in ("diagnostics", "batch", "served") else
                 2 if kind == "rows" else methods,
                 chunks=angles if kind == "chunks" else 1, pinned=kind == "host",
                 thick=rng.randint(1, 4) if kind == "thick" else 0,
                 d0=rng.uniform(0.4, 2.5) if kind == "euclid" else 0.0,
                 scans=rng.randint(3, 8) if kind in ("batch", "served") else 1)
    del case["name"]
    return case


# ------------------------------------------------------------------- inputs
def _geometry(case, scan=0):
    """The grid of a case; the scans of a batch and of a serving pass take turns at half, full and
    (in a batch) double the in-plane size."""
    f = (1.0, 0.5, 2.0)[scan % 3] if case["kind"] == "batch" else (1.0, 0.5)[scan % 2] \
        if case["kind"] == "served" else 1.0
    nx, ny = (max(8, min(256, int(case[k] * f))) if f != 1.0 else case[k] for k in ("nx", "ny"))
    T = case["T"] if f == 1.0 else math.ceil(math.hypot(nx * case["sx"], ny * case["sy"]) / 2 + 10)
    return synth.Geometry(nx, ny, case["nz"], case["sx"], case["sy"], case["sz"], float(T))


def _per_angle(case, scan=0):
    """Uneven scans: from a third of the case's histories to three times as many."""
    return case["per_angle"] if case["scans"] == 1 else \
        max(1, int(case["per_angle"] * 3.0 ** (1.0 - 2.0 * scan / (case["scans"] - 1))))


def _face(case, g):
    return (case["u_half"] or math.hypot(g.nx * g.sx, g.ny * g.sy) / 2 + 1.0,
            case["v_half"] or g.nz * g.sz / 2)


def _phantom(case, g, rng):
    hx, hy, hz = g.nx * g.sx / 2, g.ny * g.sy / 2, g.nz * g.sz / 2
    if case["phantom"] == "random":
        return synth.random_phantom(rng, g)
    if case["phantom"] == "ellipsoid":
        return [synth.Ellipsoid((0.0, 0.0, 0.0), (0.78 * hx, 0.87 * hy, 0.8 * hz), 1.0)]
    # the head phantom scaled to the volume
    return [synth.Ellipsoid(tuple(c * h / r for c, h, r in zip(e.center, (hx, hy, hz),
                                                               (100.0, 100.0, 40.0))),
                            tuple(a * h / r for a, h, r in zip(e.semi, (hx, hy, hz),
                                                               (100.0, 100.0, 40.0))), e.rsp)
            for e in synth.head_phantom()]


def _wepl(p, d, phantom):
    """RSP line integral of the segments p -> p + d through the painter's union."""
    ivs = []
    for e in phantom:
        c, a = (torch.tensor(v, dtype=torch.float32, device=p[0].device) for v in (e.center, e.semi))
        q = [(p[k] - c[k]) / a[k] for k in range(3)]
        r = [d[k] / a[k] for k in range(3)]
        A = sum(x * x for x in r)
        B = 2.0 * sum(x * y for x, y in zip(q, r))
        disc = B * B - 4.0 * A * (sum(x * x for x in q) - 1.0)
        root = disc.clamp_min(0.0).sqrt()
        ivs.append((((-B - root) / (2 * A)).clamp(0, 1), ((-B + root) / (2 * A)).clamp(0, 1)))
    zero = torch.zeros_like(d[0])
    t = torch.stack([zero, zero + 1.0] + [x for iv in ivs for x in iv]).sort(dim=0).values
    w = zero
    for k in range(len(t) - 1):
        mid, rsp = 0.5 * (t[k] + t[k + 1]), zero
        for (t0, t1), e in zip(ivs, phantom):
            rsp = torch.where((mid > t0) & (mid < t1), e.rsp, rsp)
        w = w + rsp * (t[k + 1] - t[k])
    return w * sum(x * x for x in d).sqrt()


def _histories(case, seed, scan=0):
    """Six float32 columns on the GPU (rows of one 6 x n block), grouped by gantry angle, and
    the geometry and phantom they belong to."""
    g = _geometry(case, scan)
    rng = np.random.Generator(np.random.PCG64([int(seed) & (2 ** 63 - 1), scan]))
    phantom = _phantom(case, g, rng)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(rng.integers(0, 2 ** 62)))
    U, V = _face(case, g)
    per, n_ang = _per_angle(case, scan), case["angles"]
    rows = torch.empty((6, per * n_ang), dtype=torch.float32, device="cuda")
    step = max(1, (1 << 21) // per)
    for a0 in range(0, n_ang, step):
        a1 = min(n_ang, a0 + step)
        deg = (torch.arange(a0, a1, device="cuda", dtype=torch.float32) * (360.0 / n_ang))
        deg = deg.repeat_interleave(per)
        n = deg.numel()
        uni = torch.rand((2, n), generator=gen, device="cuda")
        nor = torch.randn((3, n), generator=gen, device="cuda")
        ui, vi = (2 * uni[0] - 1) * U, (2 * uni[1] - 1) * V
        uo, vo = ui + case["sigma"] * nor[0], vi + case["sigma"] * nor[1]
        c, s = torch.cos(torch.deg2rad(deg)), torch.sin(torch.deg2rad(deg))
        p = [-g.T * c - ui * s, -g.T * s + ui * c, vi]
        q = [g.T * c - uo * s, g.T * s + uo * c, vo]
        w = _wepl(p, [y - x for x, y in zip(p, q)], phantom)
        w = w + nor[2] * (0.01 * w + 0.3)
        for k, col in enumerate((deg, ui, vi, uo, vo, w)):
            rows[k, a0 * per:a1 * per] = col
    return rows, g, phantom


def _object(g, phantom):
    """The true object as a uint8 volume (x fastest)."""
    axes = [(torch.arange(n, device="cuda", dtype=torch.float32) + 0.5 - n / 2) * s
            for n, s in ((g.nx, g.sx), (g.ny, g.sy), (g.nz, g.sz))]
    z, y, x = torch.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
    inside = torch.zeros_like(x, dtype=torch.bool)
    for e in phantom:
        inside |= sum(((v - c) / a) ** 2 for v, c, a in zip((x, y, z), e.center, e.semi)) < 1.0
    return inside.to(torch.uint8).reshape(-1)


# -------------------------------------------------------------- preparation
def _scan(case, g):
    params = H.hd_params_default()
    params.methods = case["methods"]
    scan = H.Scan(g, params)
    if case["thick"]:
        scan.set_thick(case["thick"])
    if case["d0"]:
        scan.set_thick_distance(case["d0"])
    return scan


def _volumes(case, g, host=False):
    """Where a scan's hulls and counts go: one buffer per method, and N and M."""
    V = g.nx * g.ny * g.nz
    where = dict(pin_memory=True) if host else dict(device="cuda")
    masks = {m: torch.zeros(V, dtype=torch.uint8, **where) for m in METHODS if case["methods"] & m}
    counts = {}
    if not host:
        for m in (H.HD_MSC, H.HD_SM):
            if case["methods"] & (3 if m == H.HD_MSC else 4):
                counts[m] = torch.zeros(V, dtype=torch.int32, device="cuda")
    return masks, counts


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind in ("batch", "served"):
        parts = [_histories(case, seed, k) for k in range(case["scans"])]
        state["geometry"] = [g for _, g, _ in parts]
        if kind == "batch":
            # batches run on a stream of the program's own
            state["rows"] = [[r[k] for k in range(6)] for r, _, _ in parts]
            state["scans"] = [_scan(case, g) for _, g, _ in parts]
            state["batch"] = H.Batch()
            state["stream"] = torch.cuda.Stream()
            state["out"] = [_volumes(case, g) for _, g, _ in parts]
        else:
            state["rows"] = []
            for r, _, _ in parts:
                host = torch.empty(r.shape, dtype=torch.float32, pin_memory=True)
                state["rows"].append(host.copy_(r))
            state["server"] = H.Server()
            state["params"] = H.hd_params_default()
        torch.cuda.synchronize()
        return state
    rows, g, phantom = _histories(case, seed)
    if case["pinned"]:
        rows = torch.empty(rows.shape, dtype=torch.float32, pin_memory=True).copy_(rows)
    cols = [rows[k] for k in range(6)]
    state["cols"], state["geometry"] = cols, g
    if kind == "binned":
        state["binned"] = H.Binned(g)
        state["image"] = torch.zeros(g.nx * g.ny * g.nz, dtype=torch.uint8, device="cuda")
        state["bins"] = torch.zeros(9 * state["binned"].n_bins, dtype=torch.int64, device="cuda")
        return state
    state["scan"] = scan = _scan(case, g)
    if kind == "scan":
        state["out"] = _volumes(case, g, host=case["pinned"])
        per, n = _per_angle(case), case["chunks"]
        edges = [per * (case["angles"] * k // n) for k in range(n + 1)]
        state["parts"] = [[c[a:b] for c in cols] for a, b in zip(edges, edges[1:])]
        return state
    # rows and diagnostics start from a finished scan
    scan.add(cols)
    scan.finalize()
    if kind == "rows":
        # a path has at most nx + ny + nz voxels: room for the longest in the plane
        n = rows.shape[1]
        state["csr"] = (torch.zeros(n + 1, dtype=torch.int64, device="cuda"),
                        torch.zeros(n * (g.nx + g.ny), dtype=torch.int32, device="cuda"))
    if kind == "diagnostics":
        state["out"] = _volumes(case, g)
        masks, counts = state["out"]
        for m, t in masks.items():
            scan.mask(m, out=t)
        for m, t in counts.items():
            scan.counts(m, out=t)
        state["object"] = _object(g, phantom)
        state["indices"] = torch.zeros(g.nx * g.ny * g.nz, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    return state


# --------------------------------------------------------------------- runs
def _read(scan, masks, counts, stream=None):
    for m, t in masks.items():
        scan.mask(m, out=t, stream=stream)
    for m, t in counts.items():
        scan.counts(m, out=t, stream=stream)
    return list(masks.values()) + list(counts.values())


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "scan":
        scan = state["scan"]
        scan.reset()
        for part in state["parts"]:
            scan.add(part)
        scan.finalize()
        out = _read(scan, *state["out"])
        if case["pinned"]:  # hulls on the host are read after the copies have landed
            torch.cuda.current_stream().synchronize()
        return out
    if kind == "batch":
        stream = state["stream"]
        stream.wait_stream(torch.cuda.current_stream())
        for scan, cols in zip(state["scans"], state["rows"]):
            state["batch"].add(scan, cols)
        state["batch"].run(H.HD_BATCH_RESET | H.HD_BATCH_FINALIZE, stream)
        out = [_read(scan, *vol, stream=stream) for scan, vol in zip(state["scans"], state["out"])]
        torch.cuda.current_stream().wait_stream(stream)
        return out
    if kind == "served":
        server, n = state["server"], case["angles"]
        ids = [server.open_scan(g, state["params"], n) for g in state["geometry"]]
        for k in range(n):
            for i, rows in zip(ids, state["rows"]):
                per = rows.shape[1] // n
                server.submit_rows(i, rows, k * per, per)
        out = []
        for i, g in zip(ids, state["geometry"]):
            if server.wait(i, 60_000) != H.HD_OK:
                raise RuntimeError("a served scan did not finish")
            view = server.scan(i, g)
            out.append([view.mask(m) for m in METHODS])
            server.close_scan(i)
        return out
    if kind == "binned":
        binned = state["binned"]
        binned.run(state["cols"])
        H.hd_binned_get_image(binned.handle, H.HD_BINNED_HULL, state["image"])
        H.hd_binned_get_bins(binned.handle, state["bins"])
        return [state["image"], state["bins"]]
    if kind == "rows":
        row_ptr, cols = state["csr"]
        nnz = H.hd_scan_system_rows(state["scan"].handle, H.HD_MSC, *state["cols"][:5], row_ptr,
                                    cols)
        return [nnz, row_ptr, cols]
    masks, counts = state["out"]
    g = state["geometry"]
    dims = (g.nx, g.ny, g.nz)
    filled = H.hd_fill_enclosed(masks[H.HD_MSC], dims)
    extra = [H.hd_hull_compare(h, state["object"], dims) for h in (filled, *masks.values())]
    canny = list(H.hd_sm_canny(counts[H.HD_SM], dims))
    n, indices = state["scan"].hull_indices(H.HD_MSC, state["indices"])
    return [filled, extra, canny, n, indices]


# --------------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once; one operation per voxel membership (an update of
    a count) or per history where nothing is traversed.  Uniform lines over a face of width 2U
    have a mean chord of area / 2U in the plane and cross 4 / pi voxels per voxel size."""
    nbytes = flops = 0.0
    for k in range(case["scans"]):
        g = _geometry(case, k)
        V, n = g.nx * g.ny * g.nz, _per_angle(case, k) * case["angles"]
        U, Vh = _face(case, g)
        chord = g.nx * g.sx * g.ny * g.sy / (2 * U) * min(1.0, g.nz * g.sz / (2 * Vh))
        steps = n * chord * (4 / math.pi) / math.sqrt(g.sx * g.sy)
        methods = case["methods"]
        outs = V * (bin(methods & 7).count("1") + 4 * (methods & 3 != 0) + 4 * (methods & 4 != 0))
        if case["kind"] == "scan" and case["d0"]:
            steps = max(steps, n * chord * math.pi * case["d0"] ** 2 / (g.sx * g.sy * g.sz))
        elif case["kind"] == "scan":
            steps *= 1 + 2 * case["thick"] * math.pi / 4
        if case["kind"] == "rows":  # about half of the volume lies in the hull
            nbytes += 20.0 * n + V + 8.0 * n + 4.0 * steps / 2
        elif case["kind"] == "binned":
            nbytes, steps = nbytes + 24.0 * n + V, n
        elif case["kind"] == "diagnostics":
            nbytes, steps = nbytes + 3 * V + 4 * V + 3 * V + 4 * V, V
        else:
            nbytes += 24.0 * n + (outs if case["kind"] != "served" else 3 * V)
        flops += steps
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """Every output is a whole number that has to stay equal; none has a 64-bit value."""
    return None
