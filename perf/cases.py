"""The measured workloads: what a user of the multigrid library has it do.

Sizes, faces, box edges and right-hand sides follow the workloads of ``inputs.py`` and
``bench.py`` (64^3 periodic, 256^3 Dirichlet, 512^3 mixed precision, batched and served
mixes of 32^3 to 128^3 problems, the two-level AMR solve, the ghost-fill benchmark), plus the
level operations that a user's own cycle is made of, at even, ragged and odd sizes.  Inputs
are drawn on the GPU from the seed; every pass goes through the ctypes binding ``mg``, which is
the library's Python surface.
"""
import math

import numpy as np
import torch

from paper_2403_12179_gb300 import mg

TOL = 1e-10


def listed():
    return [
        # the smallest call: one red + black sweep of one 32^3 box, as on a coarse level of a
        # user's own cycle -- four launches of a microsecond or two each
        {"name": "sweep-f64-32", "kind": "sweep", "nx": 32, "ny": 32, "nz": 32, "box": 32,
         "faces": "ppp", "dtype": "f64", "ghosts": 1, "sweeps": 1},
        # a user's own smoother loop on a large FP32 level with the two ghost layers that the
        # fused sweep wants: two full sweeps from a zero guess
        {"name": "sweep-f32-256", "kind": "sweep", "nx": 256, "ny": 256, "nz": 256, "box": 64,
         "faces": "ddd", "dtype": "f32", "ghosts": 2, "sweeps": 2},
        # residual and its norm on an odd-sized FP64 domain chopped into ragged boxes: the
        # convergence check of a user's own iteration
        {"name": "residual-f64-odd", "kind": "residual", "nx": 255, "ny": 190, "nz": 127, "box": 64,
         "faces": "ddd", "dtype": "f64"},
        # down and up between two levels: FP32 residual + restriction, then prolongation, with
        # boxes of 32^3
        {"name": "transfer-f32-192", "kind": "transfer", "nx": 192, "ny": 192, "nz": 192, "box": 32,
         "faces": "ppp", "dtype": "f32"},
        # the ghost exchange of a simulation: 4 components, 2 layers, periodic
        {"name": "fill-f64-256x4", "kind": "fill", "nx": 256, "ny": 256, "nz": 256, "box": 64,
         "faces": "ppp", "dtype": "f64", "ncomp": 4, "ghosts": 2},
        # one small solve, where launches and latency count
        {"name": "solve-f64-64", "kind": "solve", "nx": 64, "ny": 64, "nz": 64, "box": 32,
         "faces": "ppp", "precision": "f64"},
        # a domain of three different extents with mixed faces, chopped into ragged boxes
        {"name": "solve-f64-ragged", "kind": "solve", "nx": 96, "ny": 80, "nz": 112, "box": 48,
         "faces": "pdd", "precision": "f64"},
        # the benchmarked solve
        {"name": "solve-f64-256", "kind": "solve", "nx": 256, "ny": 256, "nz": 256, "box": 64,
         "faces": "ddd", "precision": "f64"},
        # the largest solve: FP32 cycles inside an FP64 iteration
        {"name": "solve-mixed-512", "kind": "solve", "nx": 512, "ny": 512, "nz": 512, "box": 128,
         "faces": "ddd", "precision": "mixed"},
        # many independent problems of several sizes, packed into shared launches
        {"name": "batch-mixed-48", "kind": "batch", "count": 48, "emin": 32, "emax": 128, "box": 32,
         "precision": "mixed"},
        # a burst of requests with their data in pinned host memory, served by the scheduler
        {"name": "serve-mixed-24", "kind": "serve", "count": 24, "emin": 32, "emax": 128, "box": 64,
         "precision": "mixed"},
        # two-level composite solve: the middle half of the domain refined
        {"name": "amr-128", "kind": "amr", "n": 128, "box": 32},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _coarsens(n, box):
    """Whether the solver takes this domain: while every extent is even and at least 4, the
    boxes have even bounds (boxes that would drop below 2 cells become one box)."""
    cuts = [[min(box, m - a) for a in range(0, m, box)] for m in n]
    while all(m % 2 == 0 and m >= 4 for m in n):
        if any(v % 2 for c in cuts for v in c):
            return False
        n = [m // 2 for m in n]
        cuts = [[v // 2 for v in c] for c in cuts]
        if any(v < 2 for c in cuts for v in c):
            cuts = [[m] for m in n]
    return n[0] * n[1] * n[2] <= 1024


def _solvable(rng, lo, hi):
    """Extents of 2 to 9 times a power of two and a box edge that coarsen, between lo and hi."""
    while True:
        k = rng.choice([3, 4, 5, 6])
        n = [rng.randint(2, 9) << k for _ in range(3)]
        if rng.random() < 0.4:
            n = [n[0]] * 3
        box = rng.choice([32, 48, 64, 128])
        if all(lo <= v <= hi for v in n) and _coarsens(n, box):
            return n, box


def _faces(rng):
    return rng.choice(["ppp", "ddd", "pdd", "dpp"])


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "residual", "transfer", "fill", "solve", "solve", "mixed",
                       "batch", "serve", "amr"])
    box = rng.choice([16, 32, 40, 64, 128])
    if kind in ("sweep", "residual", "fill"):
        n = [_spread(rng, 24, 272) for _ in range(3)]
        case = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "box": max(box, 32),
                "faces": _faces(rng), "dtype": rng.choice(["f64", "f32"])}
        if kind == "sweep":
            # (red and black need an even number of cells around a periodic direction)
            for d, f in zip(("nx", "ny", "nz"), case["faces"]):
                case[d] += case[d] % 2 if f == "p" else 0
            case["ghosts"] = rng.choice([1, 2])
            case["sweeps"] = rng.choice([1, 2])
        elif kind == "fill":
            case["ncomp"] = rng.choice([1, 1, 3, 4, 6])
            case["ghosts"] = rng.choice([1, 2, 3])
        return case
    if kind == "transfer":
        n = [2 * _spread(rng, 16, 136) for _ in range(3)]
        return {"kind": "transfer", "nx": n[0], "ny": n[1], "nz": n[2], "box": max(box, 32),
                "faces": _faces(rng), "dtype": rng.choice(["f64", "f32"])}
    if kind in ("solve", "mixed"):
        n, box = _solvable(rng, 24, 272 if kind == "solve" else 448)
        return {"kind": "solve", "nx": n[0], "ny": n[1], "nz": n[2], "box": box,
                "faces": _faces(rng), "precision": "f64" if kind == "solve" else "mixed"}
    if kind == "amr":
        return {"kind": "amr", "n": rng.choice([32, 48, 64, 80, 96, 128, 160]),
                "box": rng.choice([16, 32, 64])}
    emin = rng.choice([16, 32])
    return {"kind": kind, "count": _spread(rng, 3, 40), "emin": emin, "emax": rng.choice([48, 64, 96, 128]),
            "box": rng.choice([16, 32, 64]), "precision": rng.choice(["f64", "mixed", "mixed"])}


# ---- inputs ----------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _periodic(faces):
    return tuple(1 if c == "p" else 0 for c in faces)


def _dtype(name):
    return (mg.MG_F64, torch.float64, 8) if name == "f64" else (mg.MG_F32, torch.float32, 4)


def _centres(n):
    return (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n


def _rhs(n, periodic, g):
    """Smooth blobs plus noise, shaped (nz, ny, nx): a source term on a grid.  Fully periodic
    problems need a right-hand side of zero mean."""
    out = torch.randn(n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64) * 1e-2
    c = torch.rand(4, 3, generator=g, device="cuda", dtype=torch.float64)
    s = 0.05 + 0.1 * torch.rand(4, generator=g, device="cuda", dtype=torch.float64)
    a = torch.randn(4, generator=g, device="cuda", dtype=torch.float64)
    for k in range(4):
        e = [torch.exp(-((_centres(n[d]) - c[k, d]) ** 2) / (2 * s[k] ** 2)) for d in range(3)]
        out += (a[k] * e[2])[:, None, None] * e[1][None, :, None] * e[0][None, None, :]
    if all(periodic):
        out -= out.mean()
    return out


def _field(n, g, dtype):
    """A solution-like field: low modes plus a little noise."""
    out = torch.randn(n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64) * 1e-3
    p = torch.rand(3, 3, generator=g, device="cuda", dtype=torch.float64)
    for k in range(3):
        w = [torch.sin(2 * math.pi * ((k + 1) * _centres(n[d]) + p[k, d])) for d in range(3)]
        out += w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :] / (k + 1)
    return out.to(dtype)


class _Session:
    """A context with its own stream, and the handles a user's program keeps."""

    def __init__(self):
        self.ctx = mg.mg_init(torch.cuda.current_device())
        self.stream = torch.cuda.Stream()
        mg.mg_set_stream(self.ctx, self.stream)
        self.keep = []

    def __del__(self):
        ctx, self.ctx = self.ctx, None
        if ctx is not None:
            mg.mg_finalize(ctx)

    def boxes(self, n, box, lo=(0, 0, 0)):
        return mg.mg_box_array_create(self.ctx, lo, tuple(lo[d] + n[d] - 1 for d in range(3)), (box,) * 3)

    def fab(self, ba, dense=None, ncomp=1, ghosts=0, dtype="f64"):
        """A fab over torch memory (its storage stays alive with whatever views it)."""
        code, tdt, size = _dtype(dtype)
        nbytes = mg.mg_fab_layout(self.ctx, ba, ncomp, ghosts, code)
        mem = torch.zeros(nbytes // size + 64, dtype=tdt, device="cuda")
        skip = (-mem.data_ptr() % 256) // size
        mem = mem[skip:skip + nbytes // size]
        self.keep.append(mem)
        f = mg.mg_fab_wrap(self.ctx, ba, ncomp, ghosts, code, mem.data_ptr(), nbytes)
        if dense is not None:
            mg.mg_fab_copy_from_dense(self.ctx, f, dense.contiguous().data_ptr(), False,
                                      torch.cuda.current_stream())
            torch.cuda.current_stream().synchronize()
        return f, mem


def _options(precision):
    return mg.make_options(precision=mg.MG_PREC_MIXED if precision == "mixed" else mg.MG_PREC_F64)


def _n(case):
    return (case["nx"], case["ny"], case["nz"])


def _problems(case):
    """(edge, periodic) of every problem of a batch or burst: the edges in turn, half of the
    problems periodic and half with Dirichlet faces."""
    edges = [e for e in (16, 32, 48, 64, 96, 128) if case["emin"] <= e <= case["emax"]]
    return [(edges[i % len(edges)], (i // len(edges) + i) % 2 == 0) for i in range(case["count"])]


def _batch_rhs(case, seed):
    g = _gen(seed)
    return [_rhs((e,) * 3, (p,) * 3, g) for e, p in _problems(case)]


def prepare(case, seed):
    S = _Session()
    kind, g = case["kind"], _gen(seed)
    S.kind = kind
    if kind in ("sweep", "residual", "transfer", "fill"):
        n, per = _n(case), _periodic(case["faces"])
        S.bc, S.h = mg.make_bc(per), 1.0 / case["nx"]
        code, tdt, size = _dtype(case["dtype"])
        ba = S.boxes(n, case["box"])
        if kind == "sweep":
            S.sweeps = case["sweeps"]
            S.rhs, _ = S.fab(ba, _rhs(n, per, g).to(tdt), ghosts=case["ghosts"] - 1, dtype=case["dtype"])
            S.phi, _ = S.fab(ba, ghosts=case["ghosts"], dtype=case["dtype"])
            S.out = torch.zeros(n[2], n[1], n[0], dtype=tdt, device="cuda")
        elif kind == "residual":
            S.rhs, _ = S.fab(ba, _rhs(n, per, g).to(tdt), dtype=case["dtype"])
            S.phi, _ = S.fab(ba, _field(n, g, tdt), ghosts=1, dtype=case["dtype"])
            mg.mg_fill_boundary(S.ctx, S.phi, S.bc, torch.cuda.current_stream())
            S.r, S.out = S.fab(ba, dtype=case["dtype"])
        elif kind == "transfer":
            S.rhs, _ = S.fab(ba, _rhs(n, per, g).to(tdt), dtype=case["dtype"])
            S.phi, _ = S.fab(ba, _field(n, g, tdt), ghosts=1, dtype=case["dtype"])
            mg.mg_fill_boundary(S.ctx, S.phi, S.bc, torch.cuda.current_stream())
            S.corr, S.fine = S.fab(ba, ghosts=1, dtype=case["dtype"])
            nc = tuple(v // 2 for v in n)
            # the coarse level as a user lays it out: the fine boxes coarsened where they have
            # even bounds
            cba = S.boxes(nc, case["box"] // 2)
            S.crhs, S.coarse = S.fab(cba, dtype=case["dtype"])
            S.cphi, S.zero = S.fab(cba, ghosts=1, dtype=case["dtype"])
            S.cerr, _ = S.fab(cba, _field(nc, g, tdt), ghosts=1, dtype=case["dtype"])
        else:
            v = torch.rand(case["ncomp"], n[2], n[1], n[0], generator=g, device="cuda",
                           dtype=torch.float64).to(tdt)
            S.phi, S.out = S.fab(ba, v, ncomp=case["ncomp"], ghosts=case["ghosts"], dtype=case["dtype"])
    elif kind == "solve":
        n, per = _n(case), _periodic(case["faces"])
        S.bc, S.opt = mg.make_bc(per), _options(case["precision"])
        ba = S.boxes(n, case["box"])
        S.rhs, _ = S.fab(ba, _rhs(n, per, g), ghosts=1)
        S.phi, _ = S.fab(ba, ghosts=2)
        S.out = torch.zeros(n[2], n[1], n[0], dtype=torch.float64, device="cuda")
    elif kind == "batch":
        S.opt, S.bcs, S.rhs, S.phi, S.out = _options(case["precision"]), [], [], [], []
        for (e, p), r in zip(_problems(case), _batch_rhs(case, seed)):
            ba = S.boxes((e,) * 3, case["box"])
            S.bcs.append(mg.make_bc((p,) * 3))
            S.rhs.append(S.fab(ba, r)[0])
            S.phi.append(S.fab(ba, ghosts=1)[0])
            S.out.append(torch.zeros(e, e, e, dtype=torch.float64, device="cuda"))
    elif kind == "serve":
        S.opt, S.req = _options(case["precision"]), []
        for (e, p), r in zip(_problems(case), _batch_rhs(case, seed)):
            host = torch.empty(e, e, e, dtype=torch.float64, pin_memory=True)
            host.copy_(r)
            ans = torch.zeros(e, e, e, dtype=torch.float64, pin_memory=True)
            S.req.append((e, mg.make_bc((p,) * 3), host, ans))
        S.box = (case["box"],) * 3
    else:
        n = case["n"]
        A, B = n // 4, 3 * n // 4
        S.bc = mg.make_bc((0, 0, 0))
        ba0, ba1 = S.boxes((n,) * 3, case["box"]), S.boxes((2 * (B - A),) * 3, case["box"], (2 * A,) * 3)
        f0, f1 = _rhs((n,) * 3, (0, 0, 0), g), _rhs((2 * (B - A),) * 3, (0, 0, 0), g)
        S.rhs0, S.rhs1 = S.fab(ba0, f0)[0], S.fab(ba1, f1)[0]
        S.phi0, S.phi1 = S.fab(ba0, ghosts=1)[0], S.fab(ba1, ghosts=1)[0]
        S.out = (torch.zeros_like(f0), torch.zeros_like(f1))
    torch.cuda.synchronize()
    return S


def _told(results):
    return {"vcycles": np.array([r.vcycles for r in results]),
            "status": np.array([r.status for r in results]),
            "rel_resid": np.array([r.rel_resid for r in results])}


def run(S):
    ctx, here = S.ctx, torch.cuda.current_stream()
    if S.kind == "sweep":
        mg.mg_fab_set_val(ctx, S.phi, 0.0, True, here)
        for _ in range(S.sweeps):
            mg.mg_smooth(ctx, S.phi, S.rhs, S.bc, S.h, 2, here)
        mg.mg_fab_copy_to_dense(ctx, S.phi, S.out.data_ptr(), False, here)
        return {"phi": S.out}
    if S.kind == "residual":
        norm = mg.mg_residual(ctx, S.phi, S.rhs, S.r, S.h, True, here)
        return {"r": S.out, "norm": norm}
    if S.kind == "transfer":
        mg.mg_residual_restrict(ctx, S.phi, S.rhs, S.crhs, S.cphi, S.h, here)
        mg.mg_fab_set_val(ctx, S.corr, 0.0, True, here)
        mg.mg_prolong_add(ctx, S.cerr, S.corr, here)
        return {"coarse": S.coarse, "zero": S.zero, "fine": S.fine}
    if S.kind == "fill":
        mg.mg_fill_boundary(ctx, S.phi, S.bc, here)
        return {"fab": S.out}
    if S.kind == "serve":
        tickets = [mg.mg_submit_host(ctx, (0, 0, 0), (e - 1,) * 3, S.box, bc, rhs.data_ptr(),
                                     ans.data_ptr(), False, TOL, S.opt) for e, bc, rhs, ans in S.req]
        res = [mg.mg_poll(ctx, t)[1] for t in tickets]
        return {"phi": [q[3] for q in S.req], **_told(res)}
    s = S.stream
    s.wait_stream(here)
    if S.kind == "solve":
        mg.mg_fab_set_val(ctx, S.phi, 0.0, True, s)
        res = [mg.mg_solve(ctx, S.rhs, S.phi, S.bc, TOL, S.opt)]
        mg.mg_fab_copy_to_dense(ctx, S.phi, S.out.data_ptr(), False, s)
    elif S.kind == "batch":
        for f in S.phi:
            mg.mg_fab_set_val(ctx, f, 0.0, True, s)
        res = mg.mg_solve_batch(ctx, S.rhs, S.phi, S.bcs, TOL, S.opt)
        for f, o in zip(S.phi, S.out):
            mg.mg_fab_copy_to_dense(ctx, f, o.data_ptr(), False, s)
    else:
        for f in (S.phi0, S.phi1):
            mg.mg_fab_set_val(ctx, f, 0.0, True, s)
        res = [mg.mg_amr2_solve(ctx, S.rhs0, S.phi0, S.rhs1, S.phi1, S.bc, TOL)]
        for f, o in zip((S.phi0, S.phi1), S.out):
            mg.mg_fab_copy_to_dense(ctx, f, o.data_ptr(), False, s)
    here.wait_stream(s)
    return {"phi": S.out, **_told(res)}


# ---- what a pass cannot do without --------------------------------------------------------------

def _cycles(cells):
    """One V(2,2) cycle over all levels (8/7 of the finest): 4 sweeps of 9 operations a cell,
    residual and restriction 11, prolongation 1."""
    return cells * 8 / 7 * (4 * 9 + 11 + 1)


def work(case):
    kind = case["kind"]
    if kind == "amr":
        n = case["n"] ** 3 + (2 * (3 * case["n"] // 4 - case["n"] // 4)) ** 3
        return {"bytes": 3 * 8 * n, "flops": 11 * _cycles(n)}
    if kind in ("batch", "serve"):
        n = sum(e ** 3 for e, _ in _problems(case))
        return {"bytes": 2 * 8 * n, "flops": 9 * _cycles(n)}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "solve":
        return {"bytes": 2 * 8 * n, "flops": 9 * _cycles(n)}
    size = _dtype(case["dtype"])[2]
    if kind == "sweep":
        return {"bytes": 2 * size * n, "flops": 9 * case["sweeps"] * n}
    if kind == "residual":
        return {"bytes": 3 * size * n, "flops": 10 * n}
    if kind == "transfer":
        return {"bytes": size * (2 * n + n / 8 * 3 + n), "flops": 12 * n}
    g, c, ghosts = case["ghosts"], case["ncomp"], 0
    cuts = []
    for m in (case["nx"], case["ny"], case["nz"]):
        cuts.append([min(case["box"], m - a) for a in range(0, m, case["box"])])
    for x in cuts[0]:
        for y in cuts[1]:
            for z in cuts[2]:
                ghosts += (x + 2 * g) * (y + 2 * g) * (z + 2 * g) - x * y * z
    return {"bytes": 2 * size * c * ghosts, "flops": 0}


# ---- the same in 64 bits, in plain torch --------------------------------------------------------

def _grown(a, per, g):
    """Dense (..., nz, ny, nx) field with g ghost layers of the domain: periodic images, -mirror
    across one Dirichlet face, 0 across two or more."""
    dims = (a.dim() - 1, a.dim() - 2, a.dim() - 3)
    outside = torch.zeros((), device=a.device)
    sign = torch.ones((), dtype=a.dtype, device=a.device)
    for d in range(3):
        m = a.shape[dims[d]]
        i = torch.arange(-g, m + g, device=a.device)
        out = (i < 0) | (i >= m)
        shape = [1] * a.dim()
        shape[dims[d]] = m + 2 * g
        if per[d]:
            j = i % m
        else:
            j = torch.where(i < 0, -1 - i, torch.where(i >= m, 2 * m - 1 - i, i))
            outside = outside + out.to(torch.float32).reshape(shape)
            sign = sign * torch.where(out, -1.0, 1.0).to(a.dtype).reshape(shape)
        a = a.index_select(dims[d], j)
    return torch.where(outside > 1, torch.zeros_like(a), a * sign)


def _neighbours(p):
    c = slice(1, -1)
    return (p[c, c, :-2] + p[c, c, 2:] + p[c, :-2, c] + p[c, 2:, c] + p[:-2, c, c] + p[2:, c, c])


def _pieces(n, box):
    for z in range(0, n[2], box):
        for y in range(0, n[1], box):
            for x in range(0, n[0], box):
                yield x, y, z, min(box, n[0] - x), min(box, n[1] - y), min(box, n[2] - z)


def _storage(dense, n, box, g, size, grown=None):
    """A fab's storage (boxes x fastest, rows padded to 16 bytes, boxes to 256) with the dense
    (ncomp, nz, ny, nx) values in its valid cells, or `grown` (dense with g ghost layers, or a
    field over the whole domain) read for ghosts too."""
    parts, total = [], 0
    nc = dense.shape[0]
    q = 16 // size
    for x, y, z, a, b, c in _pieces(n, box):
        pitch = -(-(a + 2 * g) // q) * q
        buf = torch.zeros(nc, c + 2 * g, b + 2 * g, pitch, dtype=torch.float64, device="cuda")
        if grown is not None:
            buf[..., :a + 2 * g] = grown[:, z:z + c + 2 * g, y:y + b + 2 * g, x:x + a + 2 * g]
        else:
            buf[:, g:g + c, g:g + b, g:g + a] = dense[:, z:z + c, y:y + b, x:x + a]
        flat = buf.reshape(-1)
        pad = -flat.numel() % (256 // size)
        parts.append(torch.cat([flat, torch.zeros(pad, dtype=torch.float64, device="cuda")]))
    return torch.cat(parts)


def _direct(rhs, per, h):
    """The discrete solution, from the eigenvectors of each dimension's second difference;
    None for fully periodic faces (unique up to a constant only)."""
    if all(per):
        return None
    dims, vals, vecs = (2, 1, 0), [], []
    for d in range(3):
        m = rhs.shape[dims[d]]
        T = np.diag(np.full(m, -2.0)) + np.diag(np.ones(m - 1), 1) + np.diag(np.ones(m - 1), -1)
        if per[d]:
            T[0, -1] += 1.0
            T[-1, 0] += 1.0
        else:
            T[0, 0] -= 1.0
            T[-1, -1] -= 1.0
        w, v = np.linalg.eigh(T)
        vals.append(torch.from_numpy(w).cuda())
        vecs.append(torch.from_numpy(v).cuda())

    def along(a, d, m):
        return torch.tensordot(a, m, dims=([dims[d]], [0])).movedim(-1, dims[d])

    a = rhs
    for d in range(3):
        a = along(a, d, vecs[d])
    a = a / ((vals[2][:, None, None] + vals[1][None, :, None] + vals[0][None, None, :]) / (h * h))
    for d in range(3):
        a = along(a, d, vecs[d].t())
    return a.contiguous()


def exact(case, seed):
    kind, g = case["kind"], _gen(seed)
    nothing = {"vcycles": None, "status": None, "rel_resid": None}
    if kind == "amr":
        return None  # a sparse direct solve of the composite system takes minutes
    if kind in ("batch", "serve"):
        got = [_direct(r, (p,) * 3, 1.0 / e) for (e, p), r in zip(_problems(case), _batch_rhs(case, seed))]
        if all(a is None for a in got):
            return None
        if kind == "serve":
            got = [None if a is None else a.cpu() for a in got]
        return {"phi": got, **nothing}
    n, per = _n(case), _periodic(case["faces"])
    if kind == "solve":
        phi = _direct(_rhs(n, per, g), per, 1.0 / case["nx"])
        return None if phi is None else {"phi": phi, **nothing}
    code, tdt, size = _dtype(case["dtype"])
    if kind == "fill":
        v = torch.rand(case["ncomp"], n[2], n[1], n[0], generator=g, device="cuda",
                       dtype=torch.float64).to(tdt).double()
        gh = case["ghosts"]
        return {"fab": _storage(v, n, case["box"], gh, size, _grown(v, per, gh))}
    h = 1.0 / case["nx"]
    rhs = _rhs(n, per, g).to(tdt).double()
    if kind == "sweep":
        phi = torch.zeros_like(rhs)
        i = [torch.arange(m, device="cuda") for m in n]
        colour = (i[2][:, None, None] + i[1][None, :, None] + i[0][None, None, :]) % 2
        # an odd periodic extent has neighbours of one colour: the ghosts hold their values
        # from before the half-sweep, as here
        for k in range(2 * case["sweeps"]):
            new = (_neighbours(_grown(phi, per, 1)) - h * h * rhs) / 6
            phi = torch.where(colour == k % 2, new, phi)
        return {"phi": phi}
    phi = _field(n, g, tdt).double()
    r = rhs - (_neighbours(_grown(phi, per, 1)) - 6 * phi) / (h * h)
    if kind == "residual":
        return {"r": _storage(r[None], n, case["box"], 0, size), "norm": float(r.abs().max())}
    nc = tuple(v // 2 for v in n)
    coarse = r.reshape(nc[2], 2, nc[1], 2, nc[0], 2).mean(dim=(1, 3, 5))
    err = _field(nc, g, tdt).double()
    fine = err.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)
    zero = torch.zeros_like(coarse)
    return {"coarse": _storage(coarse[None], nc, case["box"] // 2, 0, size),
            "zero": _storage(zero[None], nc, case["box"] // 2, 1, size),
            "fine": _storage(fine[None], n, case["box"], 1, size)}
