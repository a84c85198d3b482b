"""Workloads of the vortex-core framework, for timing and for comparing results.

Every case is one pass through public entry points of ``paper_1911_12070_gb300``
on seeded random-wave tangles (about one pierced face per hundred nodes, the
density of the fields that the tests and the benchmark use).  A case is a dict
of plain values; ``kind`` names the path:

``step``     identification + plain localization into buffers that the caller
             keeps: the call of an in-situ loop, once per snapshot
``host``     the same from a pinned host field to host records
``stats``    identification with its face statistics (the first look at a field)
``nodes``    the paper's node form (ring circulation of every node) from psi
``refine``   sample refinement from the pierced faces' centres, then Eq. 7
``lines``    the whole vectorization of one face list: sample graph, box-mean
             reduction, line pieces, Catmull-Rom curves
``learned``  learned localization of a face list (4x4x4 encoding + network)
``train``    minibatch training steps of the learned locator from a checkpoint
``batch``    one planned pass over snapshots of different sizes

The inputs and the 64-bit values of :func:`exact` are plain torch and numpy.
"""
import functools
import math

import numpy as np
import torch

import paper_1911_12070_gb300 as qtv

DEV = "cuda"
DENSITY = 0.0105   # pierced faces per node of these tangles
WAVES = 256


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _grid_case(name, kind, nz, ny, nx, **more):
    return dict({"name": name} if name else {}, kind=kind, nz=nz, ny=ny, nx=nx, **more)


def listed():
    return [
        # the smallest grid of the tests: a live preview, where launches count
        _grid_case("step 64", "step", 64, 64, 64, noise=0.0),
        # the benchmark's step (noise leaves every phase as it was)
        _grid_case("step 512 noisy", "step", 512, 512, 512, noise=0.05),
        # a production snapshot, far larger than the L2 cache
        _grid_case("step 1024", "step", 1024, 1024, 1024, noise=0.0),
        # a cropped sub-volume: odd, ragged extents
        _grid_case("step odd", "step", 275, 301, 253, noise=0.05),
        # a field that lives on the host (read from disk, or of a CPU solver)
        _grid_case("host 256", "host", 256, 256, 256, noise=0.05),
        # how many faces are ambiguous, touch zeros or are not finite
        _grid_case("stats 256", "stats", 256, 256, 256, noise=0.05),
        # the paper's own identification (Sec. 2.2.2)
        _grid_case("nodes 384", "nodes", 384, 384, 384, noise=0.0),
        # the paper's own localization (Sec. 3.3.3) and its error measure (Eq. 7)
        _grid_case("refine 256", "refine", 256, 256, 256, noise=0.05),
        # from pierced faces to smooth curves (Sec. 3.1-3.4)
        _grid_case("lines 384", "lines", 384, 384, 384, noise=0.05),
        # noisy field, network trained for this noise
        _grid_case("learned 384", "learned", 384, 384, 384, noise=0.05),
        # a few optimizer steps at the training driver's batch size
        {"name": "train 4096", "kind": "train", "batch": 4096, "steps": 8},
        # snapshots of a run with refined grids, one pass for all
        {"name": "batch 12", "kind": "batch",
         "sizes": "128x128x128 " * 6 + "192x192x192 " * 3 + "256x256x256 " * 2 + "384x384x384"},
    ]


# smallest edge, largest edge, most nodes of a drawn grid
_RANGE = {"step": (40, 1024, 1 << 29), "host": (64, 448, 1 << 26), "stats": (64, 640, 1 << 27),
          "nodes": (64, 640, 1 << 27), "refine": (96, 448, 3 << 23), "lines": (96, 512, 1 << 26),
          "learned": (96, 512, 1 << 27)}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng, lo, hi, most, odd):
    while True:
        nz, ny, nx = (_log_int(rng, lo, hi) for _ in range(3))
        nx = nx // 2 * 2 + (1 if odd else 0)
        if nz * ny * nx <= most:
            return nz, ny, nx


def draw(rng):
    kind = rng.choice(["step", "step", "host", "stats", "nodes", "refine", "lines", "learned",
                       "train", "batch"])
    if kind == "train":
        return {"kind": kind, "batch": 64 * _log_int(rng, 4, 128), "steps": rng.randint(4, 8)}
    if kind == "batch":
        n = rng.randint(3, 16)
        shapes = [_draw_shape(rng, 64, 320, 1 << 23, False) for _ in range(n)]
        return {"kind": kind, "sizes": " ".join("%dx%dx%d" % s for s in shapes)}
    lo, hi, most = _RANGE[kind]
    nz, ny, nx = _draw_shape(rng, lo, hi, most, rng.random() < 1 / 3)
    noise = rng.choice([0.0, 0.05]) if kind in ("step", "nodes") else 0.05
    return _grid_case(None, kind, nz, ny, nx, noise=noise)


def work(case):
    """Each input read once and each output written once."""
    if case["kind"] == "train":
        rows = case["batch"] * case["steps"]
        # forward, data gradient (not of the first layer) and weight gradient
        flops = 2 * rows * (3 * 99072 - 128 * 256)
        return {"bytes": rows * (256 + 12) + 6 * 4 * qtv.LOCATOR_PARAMS, "flops": flops}
    if case["kind"] == "batch":
        n = sum(math.prod(s) for s in _sizes(case))
    else:
        n = case["nz"] * case["ny"] * case["nx"]
    f = DENSITY * n
    # field 8, face 8 + 1, sample 12 + 4 + 1 bytes
    by = {"step": 8 * n + 26 * f, "batch": 8 * n + 26 * f, "host": 8 * n + 32 * f,
          "stats": 8 * n + 9 * f, "nodes": 8 * n + 0.025 * n * 11,
          # faces, then points, densities, tangents, determinants, steps, flags; mean density
          "refine": 8 * n + f * (8 + 37),
          # faces with samples; neighbours, degrees, labels twice, means, node lists, curves
          "lines": f * (21 + 45 + 4 + 24 + 4 + 96),
          "learned": 8 * n + 26 * f}[case["kind"]]
    return {"bytes": by, "flops": f * 198144 if case["kind"] == "learned" else 0}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _field(shape, seed, noise, waves=WAVES):
    """psi = sum of plane waves, |k| uniform in [0.15, 0.35] rad / h, complex
    Gaussian amplitudes, mean |psi|^2 = 1; times (1 + noise g), g real normal."""
    nz, ny, nx = shape
    gen = torch.Generator().manual_seed(int(seed))
    d = torch.randn(waves, 3, generator=gen, dtype=torch.float64)
    k = d / d.norm(dim=1, keepdim=True) * (0.15 + 0.2 * torch.rand(waves, 1, generator=gen,
                                                                    dtype=torch.float64))
    amp = torch.complex(torch.randn(waves, generator=gen, dtype=torch.float64),
                        torch.randn(waves, generator=gen, dtype=torch.float64))
    amp = (amp * math.sqrt(0.5 / waves)).to(DEV)
    k = k.to(DEV)

    def table(axis, n):
        ph = torch.outer(k[:, axis], torch.arange(n, dtype=torch.float64, device=DEV))
        return torch.polar(torch.ones_like(ph), ph).to(torch.complex64)

    ex, ey = table(0, nx), table(1, ny).T.contiguous()          # [W, nx], [ny, W]
    ez = (table(2, nz) * amp[:, None].to(torch.complex64)).T    # [nz, W]
    psi = torch.empty(shape, dtype=torch.complex64, device=DEV)
    step = max(1, (1 << 26) // (ny * waves))
    for z in range(0, nz, step):
        m = ez[z:z + step, None, :] * ey[None]
        torch.matmul(m.reshape(-1, waves), ex, out=psi[z:z + step].view(-1, nx))
    if noise:
        _noise(psi, seed, noise)
    return psi


def _noise(psi, seed, level):
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 100000)
    for plane in psi:
        plane *= 1 + level * torch.randn(plane.shape, generator=gen, device=DEV)


def _case_field(case, seed):
    """The field of a case.  The paths whose results are lists as long as what
    they find take a fixed tangle, mirrored, conjugated and with amplitude noise
    by the seed: other positions and faces, but as many."""
    shape = case["nz"], case["ny"], case["nx"]
    if case["kind"] in ("step", "nodes"):
        return _field(shape, seed, case["noise"])
    psi = _field(shape, 7, 0.0)
    gen = torch.Generator().manual_seed(int(seed))
    bits = torch.randint(2, (4,), generator=gen).tolist()
    psi = psi.flip([d for d in range(3) if bits[d]])
    if bits[3]:
        psi = psi.conj().resolve_conj()
    _noise(psi, seed, case["noise"])
    return psi


def _faces(psi):
    """Pierced faces of psi by the wrapped phase differences in 64 bits: ids
    ascending (linear index of the minimum corner * 4 + orientation; 0 = xy,
    1 = yz, 2 = zx) and windings."""
    nz, ny, nx = psi.shape
    tau = 2 * math.pi

    def wrap(d):
        return d - tau * torch.ceil(d / tau - 0.5)

    ids, ws = [], []
    step = max(1, (1 << 24) // (ny * nx))
    for z in range(0, nz, step):
        n = min(step, nz - z)  # planes whose faces are listed here
        ph = torch.angle(psi[z:z + n + 1].to(torch.complex128))
        dx = wrap(ph[:, :, 1:] - ph[:, :, :-1])
        dy = wrap(ph[:, 1:] - ph[:, :-1])
        dz = wrap(ph[1:] - ph[:-1])
        loops = (dx[:n, :-1] + dy[:n, :, 1:] - dx[:n, 1:] - dy[:n, :, :-1],
                 dy[:-1] + dz[:, 1:] - dy[1:] - dz[:, :-1],
                 dz[:, :, :-1] + dx[1:] - dz[:, :, 1:] - dx[:-1])
        part, wpart = [], []
        for o, c in enumerate(loops):
            w = torch.round(c / tau)
            at = torch.nonzero(w, as_tuple=True)
            part.append((((at[0] + z) * ny + at[1]) * nx + at[2]) * 4 + o)
            wpart.append(w[at].to(torch.int8))
        part, wpart = torch.cat(part), torch.cat(wpart)
        part, order = torch.sort(part)
        ids.append(part)
        ws.append(wpart[order])
    return torch.cat(ids), torch.cat(ws)


def _split(ids, shape):
    """Orientation and minimum corner (x, y, z) of faces."""
    nz, ny, nx = shape
    lin = ids >> 2
    return ids & 3, torch.stack([lin % nx, lin // nx % ny, lin // (nx * ny)], 1)


def _frame(o, shape, strides=False):
    """Per face its axes (u, v, n) as 0 = x, 1 = y, 2 = z, or their strides."""
    ax = torch.tensor([[0, 1, 2], [1, 2, 0], [2, 0, 1]], device=o.device)
    if not strides:
        return ax[o]
    return torch.tensor([1, shape[2], shape[1] * shape[2]], device=o.device)[ax[o]]


def _zeros(psi, ids):
    """(u, v) of the bilinear interpolant's zero on each face, in 64 bits."""
    o, _ = _split(ids, psi.shape)
    st = _frame(o, psi.shape, strides=True)
    flat, lin = psi.reshape(-1), ids >> 2
    p0, p1, p2, p3 = (flat[lin + off].to(torch.complex128)
                      for off in (0, st[:, 0], st[:, 0] + st[:, 1], st[:, 1]))
    a, b, c, d = p0, p1 - p0, p3 - p0, p2 - p1 - p3 + p0

    def cross(p, q):
        return (p * q.conj()).imag

    # u = -(a + c v) / (b + d v) is real: a quadratic in v
    q2, q1, q0 = cross(c, d), cross(a, d) + cross(c, b), cross(a, b)
    s = -0.5 * (q1 + torch.copysign(torch.sqrt(torch.clamp(q1 * q1 - 4 * q2 * q0, min=0)), q1))
    v = torch.stack([s / q2, q0 / s])
    p, q = a + c * v, b + d * v
    u = -(p * q.conj()).real / (q.abs() ** 2)
    out = torch.maximum((u - 0.5).abs(), (v - 0.5).abs())
    best = torch.nan_to_num(out, nan=1e300).argmin(0, keepdim=True)
    return torch.stack([u.gather(0, best)[0], v.gather(0, best)[0]], 1)


def _positions(ids, uv, shape):
    o, corner = _split(ids, shape)
    ax = _frame(o, shape)
    return corner.double().scatter_add(1, ax[:, :2], uv)


def _encode(psi, ids, w, dtype=torch.float64):
    """The learned locator's input: the 4x4x4 block around each face in the
    face frame, conjugated for W = -1, rotated by the minimum corner's phase,
    divided by the block's RMS.  (x [n, 128], inside the grid, rms)."""
    nz, ny, nx = psi.shape
    o, corner = _split(ids, psi.shape)
    top = torch.tensor([nx, ny, nz], device=ids.device)
    ok = ((corner >= 1) & (corner + 2 < top)).all(1)
    st = _frame(o, psi.shape, strides=True)
    r = torch.arange(-1, 3, device=ids.device)
    off = (st[:, 2, None, None, None] * r[:, None, None] + st[:, 1, None, None, None] * r[:, None]
           + st[:, 0, None, None, None] * r)
    at = ((ids >> 2)[:, None] + off.reshape(-1, 64)).clamp(0, psi.numel() - 1)
    cplx = torch.complex128 if dtype == torch.float64 else torch.complex64
    p = psi.reshape(-1)[at].to(cplx)
    p = torch.where((w == -1)[:, None], p.conj(), p)
    p = p * (p[:, 21:22].conj() / p[:, 21:22].abs())
    rms = (p.abs() ** 2).mean(1).sqrt()
    return torch.view_as_real(p / rms[:, None]).reshape(-1, 128), ok, rms


def _layers(flat):
    """W1, b1, W2, b2, W3, b3 of the flat parameter vector."""
    sizes = [(256, 128), (256,), (256, 256), (256,), (3, 256), (3,)]
    parts = torch.split(flat, [math.prod(s) for s in sizes])
    return [p.view(s) for p, s in zip(parts, sizes)]


def _network(flat, x):
    w1, b1, w2, b2, w3, b3 = _layers(flat)
    return torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3.T + b3


def _initial(seed):
    gen = torch.Generator().manual_seed(int(seed))
    flat = torch.zeros(qtv.LOCATOR_PARAMS)
    for m in _layers(flat)[::2]:
        m.copy_(torch.randn(m.shape, generator=gen) * math.sqrt(2 / m.shape[1]))
    return flat.to(DEV)


def _adam(flat, m, v, t, lr, grad):
    m.mul_(0.9).add_(grad, alpha=0.1)
    v.mul_(0.999).addcmul_(grad, grad, value=0.001)
    flat.sub_(lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8))


def _examples(seed, n):
    """Encodings (FP32) of a noisy n^3 field's faces and the clean zeros."""
    clean = _field((n, n, n), seed, 0.0)
    ids, w = _faces(clean)
    x, ok, _ = _encode(_field((n, n, n), seed, 0.05), ids, w, torch.float32)
    uv = _zeros(clean, ids)
    t = torch.cat([uv, torch.zeros_like(uv[:, :1])], 1).float()
    return x[ok].contiguous(), t[ok].contiguous()


@functools.lru_cache(maxsize=1)
def _trained():
    """Weights of a short training in plain torch: what a user has on disk."""
    x, t = _examples(101, 160)
    flat = _initial(1)
    m, v = torch.zeros_like(flat), torch.zeros_like(flat)
    gen = torch.Generator().manual_seed(1)
    steps, batch = 600, 4096
    for s in range(1, steps + 1):
        at = torch.randint(x.shape[0], (batch,), generator=gen).to(DEV)
        p = flat.clone().requires_grad_(True)
        loss = (_network(p, x[at]) - t[at]).square().sum(1).mean()
        grad, = torch.autograd.grad(loss, p)
        _adam(flat, m, v, s, 2e-3 * 0.5 * (1 + math.cos(math.pi * s / steps)) + 1e-5, grad)
    return flat.cpu()


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split()]


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _capacity(n):
    return max(1024, int(0.02 * n))


def _outputs(cap):
    return {"ids": torch.zeros(cap, dtype=torch.int64, device=DEV),
            "w": torch.zeros(cap, dtype=torch.int8, device=DEV),
            "xyz": torch.zeros((cap, 3), device=DEV), "resid": torch.zeros(cap, device=DEV),
            "flags": torch.zeros(cap, dtype=torch.uint8, device=DEV)}


def _train_inputs(case, seed):
    """Rows of `steps` minibatches (BF16), their targets and a fresh network."""
    x, t = _examples(seed, 128)
    gen = torch.Generator().manual_seed(int(seed))
    at = torch.randint(x.shape[0], (case["steps"], case["batch"]), generator=gen).to(DEV)
    return x[at].to(torch.bfloat16), t[at], _initial(seed)


RATE = 1e-3
BOX = 4.0


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "q": qtv.Qtv(0)}
    if kind == "train":
        x, t, flat = _train_inputs(case, seed)
        s.update(x=[r.view(torch.int16).contiguous() for r in x], t=[r.contiguous() for r in t],
                 params=flat.cpu().numpy(), adam=np.zeros(2 * flat.numel(), np.float32),
                 loss=torch.zeros(case["steps"], device=DEV))
        s["q"].locator_set(s["params"], s["adam"], 0)
        return s
    if kind == "batch":
        s["psis"] = [_field(n, seed * 64 + i, 0.0) for i, n in enumerate(_sizes(case))]
        s["q"].batch_plan(s["psis"])
        s["out"] = _outputs(_capacity(sum(p.numel() for p in s["psis"])))
        s["offsets"] = torch.zeros(len(s["psis"]) + 1, dtype=torch.int64, device=DEV)
        return s
    shape = _shape(case)
    n = math.prod(shape)
    psi = _case_field(case, seed)
    if kind == "host":
        s["psi"] = psi.cpu().pin_memory()
        return s
    s["psi"] = psi
    if kind == "step":
        s["out"] = _outputs(_capacity(n))
        s["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        s["q"].reserve(shape, _capacity(n))
    elif kind == "nodes":
        cap = max(1024, int(0.06 * n))
        s["ids"] = torch.zeros(cap, dtype=torch.int64, device=DEV)
        s["circ"] = torch.zeros((cap, 3), dtype=torch.int8, device=DEV)
        s["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    elif kind in ("refine", "lines", "learned"):
        s["ids"], s["w"] = _faces(psi)
        if kind == "lines":
            s["xyz"] = _positions(s["ids"], _zeros(psi, s["ids"]), shape).float()
            s["shape"] = shape
            s["means"] = torch.zeros((s["ids"].numel(), 3), dtype=torch.float64, device=DEV)
            del s["psi"]
        elif kind == "learned":
            s["q"].locator_set(_trained().numpy())
            s["out"] = _outputs(s["ids"].numel())
    return s


def run(s):
    kind, q = s["kind"], s["q"]
    if kind == "step":
        o = s["out"]
        q.identify_localize_into(s["psi"], o["ids"], o["w"], s["count"], o["xyz"], o["resid"],
                                 o["flags"])
        return {"count": s["count"], **o}
    if kind == "host":
        r = q.identify_localize_host(s["psi"])
        return {f: r[f] for f in ("x", "y", "z", "resid", "face_id", "winding", "flags")}
    if kind == "stats":
        ids, w, st = q.identify(s["psi"], stats=True)
        return {"ids": ids, "w": w, "stats": st}
    if kind == "nodes":
        q.node_circulation_into(s["psi"], s["ids"], s["circ"], s["count"])
        return {"ids": s["ids"], "circ": s["circ"], "count": s["count"]}
    if kind == "refine":
        out = q.refine_samples(s["psi"], face_ids=s["ids"])
        e, mean_rho, rho_bar = q.density_error(s["psi"], out["xyz"])
        return {**out, "e": e, "mean_rho": mean_rho, "rho_bar": rho_bar}
    if kind == "lines":
        nbr, deg, comp, ncomp = q.face_graph(s["shape"], s["ids"])
        label, reps, means, passes = q.box_reduce(nbr, deg, s["xyz"], box=BOX)
        s["means"].index_copy_(0, reps, means)  # at each cluster's lowest sample
        pieces, nodes = q.line_pieces(nbr, deg, comp, s["xyz"], s["ids"], s["w"])
        curve, first, length = q.piece_curves(s["xyz"], nodes, pieces)
        return {"nbr": nbr, "deg": deg, "comp": comp, "ncomp": ncomp, "label": label,
                "means": s["means"], "passes": passes, "pieces": pieces,
                "nodes": nodes, "curve": curve, "first": first, "length": length}
    if kind == "learned":
        o = s["out"]
        q.localize_into(s["psi"], s["ids"], s["w"], o["xyz"], o["resid"], o["flags"],
                        mode=qtv.LEARNED)
        return {f: o[f] for f in ("xyz", "resid", "flags")}
    if kind == "train":
        q.locator_set(s["params"], s["adam"], 0)
        for i, (x, t) in enumerate(zip(s["x"], s["t"])):
            q.locator_train_step(x, t, RATE, loss=s["loss"][i:i + 1])
        params, adam, step = q.locator_get()
        return {"loss": s["loss"], "params": params, "adam": adam, "step": step}
    o = s["out"]
    q.batch_run_into(o["ids"], o["w"], s["offsets"], o["xyz"], o["resid"], o["flags"])
    return {"offsets": s["offsets"], **o}


# ---------------------------------------------------------------------------
# 64-bit values (None: whole numbers, or a residual that is zero up to rounding)
# ---------------------------------------------------------------------------
def _padded(rows, cap):
    out = torch.zeros((cap, 3), dtype=torch.float64, device=DEV)
    out[:rows.shape[0]] = rows
    return out


def _plain(psi):
    ids, _ = _faces(psi)
    return _positions(ids, _zeros(psi, ids), psi.shape)


def _tangents(psi, ids):
    """Unit pseudo-vorticity grad Re psi x grad Im psi at the face centres:
    trilinear means of central node differences (one-sided on the boundary)."""
    shape = psi.shape
    o, corner = _split(ids, shape)
    mid = corner.double().scatter_add(1, _frame(o, shape)[:, :2],
                                      torch.full((ids.numel(), 2), 0.5, dtype=torch.float64,
                                                 device=DEV))
    top = torch.tensor(shape[::-1], device=DEV) - 1
    cell = torch.minimum(mid.floor().long(), top - 1)
    f = mid - cell
    flat = psi.reshape(-1)

    def at(p):
        return flat[(p[:, 2] * shape[1] + p[:, 1]) * shape[2] + p[:, 0]].to(torch.complex128)

    g = torch.zeros((ids.numel(), 3), dtype=torch.complex128, device=DEV)
    for n in range(8):
        bit = torch.tensor([n & 1, n >> 1 & 1, n >> 2], device=DEV)
        weight = torch.where(bit.bool(), f, 1 - f).prod(1)
        for axis in range(3):
            e = torch.zeros(3, dtype=torch.long, device=DEV)
            e[axis] = 1
            hi = torch.minimum(cell + bit + e, top)
            lo = (cell + bit - e).clamp(min=0)
            g[:, axis] += weight * (at(hi) - at(lo)) / (hi - lo)[:, axis]
    t = torch.linalg.cross(g.real, g.imag)
    return t / t.norm(dim=1, keepdim=True)


def _walks(ids, w, xyz, shape):
    """Ordered line pieces of the faces' graph (two faces are neighbours when
    they bound the same cell): [(sample indices, closed)] in the documented order."""
    nz, ny, nx = shape
    o, corner = (t.cpu().numpy() for t in _split(ids, shape))
    p, n = xyz.double().cpu().numpy(), ids.numel()
    axis = np.array([2, 0, 1])[o]                      # each face's normal
    low = corner.copy()
    low[np.arange(n), axis] -= 1                       # the cell on its other side
    cell, face = np.concatenate([corner, low]), np.tile(np.arange(n), 2)
    ok = ((cell >= 0) & (cell < np.array([nx, ny, nz]) - 1)).all(1)
    cell, face = cell[ok], face[ok]
    key = (cell[:, 2] * ny + cell[:, 1]) * nx + cell[:, 0]
    order = np.argsort(key, kind="stable")
    key, face = key[order], face[order]
    pairs = [np.stack([face[:-d], face[d:]], 1)[key[:-d] == key[d:]] for d in range(1, 6)]
    pairs = np.concatenate(pairs)
    pairs = np.concatenate([pairs, pairs[:, ::-1]])
    pairs = pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))]
    start = np.searchsorted(pairs[:, 0], np.arange(n + 1)).tolist()
    to = pairs[:, 1].tolist()
    adj = [to[start[i]:start[i + 1]] for i in range(n)]
    seen, found = [False] * n, []

    def walk(b, v, stop):
        path, prev, cur = [b, v], b, v
        while cur not in stop:
            nb = [q for q in adj[cur] if q != prev]
            if not nb:
                break
            prev, cur = cur, nb[0]
            if cur == b:
                return path, True
            path.append(cur)
        return path, False

    for i in range(n):
        if seen[i]:
            continue
        comp, todo = [], [i]
        seen[i] = True
        while todo:
            c = todo.pop()
            comp.append(c)
            for q in adj[c]:
                if not seen[q]:
                    seen[q] = True
                    todo.append(q)
        branch = sorted(c for c in comp if len(adj[c]) > 2)
        ends = [c for c in comp if len(adj[c]) == 1]
        if len(comp) == 1:
            found.append((comp, False))
        elif branch:
            used, stop = set(), set(branch)
            for b in branch:
                for v in adj[b]:
                    if (b, v) not in used:
                        path, closed = walk(b, v, stop)
                        used.update([(b, v), (path[-1], b if closed else path[-2])])
                        found.append((path, closed))
        else:
            first = min(ends) if ends else i
            found.append(walk(first, adj[first][0], set()))
    found.sort(key=lambda f: (f[0][0], f[0][1] if len(f[0]) > 1 else -1))
    d = np.zeros((n, 3))
    d[np.arange(n), axis] = w.cpu().numpy()
    out = []
    for path, closed in found:
        q = p[path + path[:1] if closed else path]
        if len(path) > 1 and np.sum(np.diff(q, axis=0) * d[path][:len(q) - 1]) < 0:
            path = path[:1] + path[:0:-1] if closed else path[::-1]
        out.append((path, closed))
    return out, p


def _curves(walks, p, per):
    """Uniform Catmull-Rom points of every piece, piece by piece, and lengths."""
    t = np.arange(per)[:, None] / per
    points, lengths = [], []
    for path, closed in walks:
        q = p[path]
        if len(q) > 1:
            e = np.vstack([q[-1:], q, q[:2]] if closed else [q[:1], q, q[-1:]])
            a, b, c, d = (e[k:len(e) - 3 + k, None] for k in range(4))
            m = 0.5 * (2 * b + t * (c - a) + t ** 2 * (2 * a - 5 * b + 4 * c - d)
                       + t ** 3 * (3 * b - a - 3 * c + d))
            q = np.vstack([m.reshape(-1, 3)] + ([] if closed else [q[-1:]]))
        points.append(q)
        r = np.vstack([q, q[:1]]) if closed else q
        lengths.append(np.sqrt((np.diff(r, axis=0) ** 2).sum(1)).sum())
    return torch.from_numpy(np.concatenate(points)), torch.tensor(lengths, dtype=torch.float64)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, flat = _train_inputs(case, seed)
        flat, t = flat.double(), t.double()
        m, v = torch.zeros_like(flat), torch.zeros_like(flat)
        losses = []
        for s in range(case["steps"]):
            p = flat.clone().requires_grad_(True)
            loss = (_network(p, x[s].double()) - t[s]).square().sum(1).mean()
            grad, = torch.autograd.grad(loss, p)
            losses.append(loss.detach())
            _adam(flat, m, v, s + 1, RATE, grad)
        return {"loss": torch.stack(losses), "params": flat, "adam": torch.cat([m, v]),
                "step": None}
    if kind == "batch":
        rows = torch.cat([_plain(_field(n, seed * 64 + i, 0.0))
                          for i, n in enumerate(_sizes(case))])
        return {"offsets": None, "ids": None, "w": None, "resid": None, "flags": None,
                "xyz": _padded(rows, _capacity(sum(math.prod(n) for n in _sizes(case))))}
    if kind in ("stats", "nodes"):
        return None  # whole numbers only
    shape = _shape(case)
    psi = _case_field(case, seed)
    if kind == "step":
        return {"count": None, "ids": None, "w": None, "resid": None, "flags": None,
                "xyz": _padded(_plain(psi), _capacity(math.prod(shape)))}
    if kind == "host":
        p = _plain(psi)
        return {"x": p[:, 0], "y": p[:, 1], "z": p[:, 2], "resid": None, "face_id": None,
                "winding": None, "flags": None}
    ids, w = _faces(psi)
    if kind == "refine":
        # the search has no closed form; its plane's normal and the mean density do
        rho_bar = sum(float((z.to(torch.complex128).abs() ** 2).sum()) for z in psi) / psi.numel()
        return {"xyz": None, "rho": None, "t": _tangents(psi, ids), "detj": None, "iters": None,
                "flags": None, "e": None, "mean_rho": None, "rho_bar": rho_bar}
    uv = _zeros(psi, ids)
    if kind == "lines":
        # the means are fixed-point sums: they are exact as they stand
        curve, length = _curves(*_walks(ids, w, _positions(ids, uv, shape).float(), shape), 8)
        return {"nbr": None, "deg": None, "comp": None, "ncomp": None, "label": None,
                "means": None, "passes": None, "pieces": None, "nodes": None,
                "curve": curve, "first": None, "length": length}
    flat = _trained().double().to(DEV)
    for a in range(0, ids.numel(), 1 << 18):
        part = slice(a, a + (1 << 18))
        x, ok, rms = _encode(psi, ids[part], w[part])
        y = _network(flat, torch.nan_to_num(x))[:, :2]
        o, _ = _split(ids[part], shape)
        st = _frame(o, shape, strides=True)
        at, (u, v) = ids[part] >> 2, y.T
        p = [psi.reshape(-1)[(at + off).clamp(max=psi.numel() - 1)].to(torch.complex128)
             for off in (0, st[:, 0], st[:, 0] + st[:, 1], st[:, 1])]
        f = (1 - u) * (1 - v) * p[0] + u * (1 - v) * p[1] + u * v * p[2] + (1 - u) * v * p[3]
        use = ok & (y >= -0.01).all(1) & (y <= 1.01).all(1) & (f.abs() ** 2 <= 1e-3 * rms ** 2)
        uv[part] = torch.where(use[:, None], y, uv[part])
    return {"xyz": _positions(ids, uv, shape), "resid": None, "flags": None}
