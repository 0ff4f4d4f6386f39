"""What a planning program has this library do, as cases that can be timed and compared.

The inputs are re-planning problems made on the GPU from a seed: an elliptic body
with a target, a margin around it and organs at risk, whose places and sizes
move with the seed as a patient's do from day to day, unspecified tissue down-sampled
2 x 2 x 2, and a dose-deposition matrix D from a parallel pencil-beam model with a
1 % jitter.  The sizes are those of this repository's workloads (the small box, the
prostate-shaped and the head-and-neck-shaped plans); ``draw`` spreads over the
ranges they span.

kinds of case (one pass each):
  plan     column generation from an empty pool on a resident D, and the plan read back
  batch    the same for several patients in one call
  import   a saved aperture pool taken over on a resident D: columns, master solve, dose
  replan   the whole of a warm-started re-plan from host arrays: upload and device build,
           the saved pool, the dose back to the host, the context released
  price    the pricing sub-problem at the current master optimum
  dose     dose, gradient and objective of a fluence (the forward product)
  prices   the beamlet prices of a dual (the transposed product)
  noalloc  dose, gradient and objective without a context or an allocation

Objectives, reduced costs and intensities come out of FP32 products, so they are
handed on as FP32, like the doses.  Intensities have no exact value: where the
optimum is flat, several pools of intensities give the same dose and objective.
"""
import functools
import math
import types

import numpy as np
import torch

import paper_1003_5402_gb300.binding as dao

DEV = "cuda"
VOXEL, BEAMLET, SIGMA, MU, CUT = 2.5, 5.0, 3.0, 0.005, 1e-3   # mm, mm, mm, 1 / mm, of a beamlet's largest entry
PREC = {"fp32": dao.DAO_PREC_FP32, "fp16": dao.DAO_PREC_FP16, "bf16": dao.DAO_PREC_BF16}
VALUE_BYTES = {"fp32": 4, "fp16": 2, "bf16": 2}

HN = dict(nx=192, ny=160, nz=80, down=True, beams=5, rows=30, cols=30)
PROSTATE = dict(nx=200, ny=120, nz=60, down=True, beams=9, rows=20, cols=20)
SMALL = dict(nx=40, ny=40, nz=12, down=False, beams=5, rows=10, cols=10)


def listed():
    def case(name, kind, size, storage, apertures, **more):
        return dict(name=name, kind=kind, **size, storage=storage, apertures=apertures,
                    **{"mlc": "consecutive", "voxelwise": False, "plans": 1, **more})
    return [
        # the headline: one head-and-neck-shaped plan of 50 apertures, mixed-precision storage
        case("plan_hn_fp16", "plan", HN, "fp16", 50),
        # a small field, planned while somebody waits: latency and launches count
        case("plan_small_fp32", "plan", SMALL, "fp32", 20),
        # a clinic's morning: several patients' plans in one call
        case("batch_prostate_fp16", "batch", PROSTATE, "fp16", 20, plans=8),
        # the online re-plan: yesterday's apertures on today's anatomy, D from the host
        case("replan_prostate_fp32", "replan", PROSTATE, "fp32", 20),
        # the saved pool re-weighted on a D that is resident already
        case("import_hn_bf16", "import", HN, "bf16", 40),
        # one pricing step of a program that drives column generation itself
        case("price_hn_fp16", "price", HN, "fp16", 12),
        # the same for an MLC whose leaves may not interdigitate
        case("price_prostate_interdig", "price", PROSTATE, "fp32", 12, mlc="interdigitation"),
        # forward product: each evaluation of a fluence by a program with its own optimiser
        case("dose_hn_fp16", "dose", HN, "fp16", 10),
        case("dose_small_fp32", "dose", SMALL, "fp32", 10),
        # the same with the re-optimisation mode's weights and thresholds per voxel
        case("dose_prostate_voxelwise", "dose", PROSTATE, "fp32", 18, voxelwise=True),
        # transposed product: the other half of such an optimiser's gradient
        case("prices_hn_fp32", "prices", HN, "fp32", 10),
        # the caller that must not allocate while a fraction runs
        case("noalloc_hn_fp32", "noalloc", HN, "fp32", 10),
    ]


def draw(rng):
    kind = rng.choice(["plan", "batch", "import", "replan", "price", "dose", "prices", "noalloc"])
    edge = int(round(math.exp(rng.uniform(math.log(36), math.log(196)))))
    down = edge >= 90
    nx, ny, nz = edge, int(edge * rng.uniform(0.6, 0.85)), max(12, int(edge * rng.uniform(0.28, 0.42)))
    if down:
        nx, ny, nz = nx // 2 * 2, ny // 2 * 2, nz // 2 * 2
    side = lambda: int(round(max(8, min(30, edge * VOXEL / BEAMLET * rng.uniform(0.22, 0.4)))))
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, down=down, beams=rng.choice([3, 4, 5, 7, 9]), rows=side(), cols=side(),
             storage=rng.choice(["fp32", "fp16", "bf16"]) if kind != "noalloc" else "fp32",
             apertures=rng.randint(5, 40 if kind in ("import", "replan") else 20),
             mlc=rng.choice(["consecutive"] * 3 + ["interdigitation"]) if kind == "price" else "consecutive",
             voxelwise=kind in ("dose", "import") and rng.random() < 0.3,
             plans=rng.randint(2, 6) if kind == "batch" else 1)
    c["beams"] = min(c["beams"], 5) if edge > 170 else c["beams"]
    return c


# ---- the problem ------------------------------------------------------------------

def _unit(seed, n):
    """n numbers in [0, 1) of a seed, on the host."""
    return np.random.default_rng(seed).random(n)


def _ellipsoid(g, centre, radii):
    return sum(((x - c) / r) ** 2 for x, c, r in zip(g, centre, radii)) <= 1.0


def _anatomy(case, seed):
    """Voxel centres (mm), the structure of each (0 target, 1 margin, 2.. organs at risk, last: body)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ax = [(torch.arange(n, device=DEV, dtype=torch.float64) + 0.5 - 0.5 * n) * VOXEL for n in (nx, ny, nz)]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")     # stored by slices, as a CT is
    h = [0.5 * n * VOXEL for n in (nx, ny, nz)]
    u = _unit((seed, 1), 16)
    at = [2.0 * (2 * u[k] - 1) for k in range(3)]                    # the day's shift, mm
    inside = (x / (0.98 * h[0])) ** 2 + (y / (0.98 * h[1])) ** 2 <= 1.0
    r = min(h[0] * 0.22, h[1] * 0.28, h[2] * 0.6, 0.45 * min(case["rows"], case["cols"]) * BEAMLET)
    organs = [((0.0, -1.35 * r, 0.0), (0.35 * r, 0.35 * r, 2.0 * r)), ((1.5 * r, 0.2 * r, 0.3 * r), (0.45 * r, 0.6 * r, 0.6 * r)),
              ((-1.5 * r, 0.2 * r, 0.3 * r), (0.45 * r, 0.6 * r, 0.6 * r))]
    grow = lambda c, rad, f, mm=0.0: _ellipsoid((x, y, z), c, [f * v + mm for v in rad])
    shapes = [grow(at, (0.55 * r, 0.5 * r, 0.6 * r), 1.0), grow(at, (r, 0.9 * r, r), 1.0)]
    shapes += [grow(c, rad, 0.9 + 0.2 * u[3 + k]) for k, (c, rad) in enumerate(organs)]   # the day's size of each organ
    body = len(shapes)
    lab = torch.full(x.shape, body, device=DEV, dtype=torch.int32)
    for k in reversed(range(body)):
        lab[shapes[k]] = k
    # full resolution wherever a structure may lie on any day
    region = functools.reduce(torch.logical_or, [grow(c, rad, 1.1) for c, rad in organs],
                              grow((0.0, 0.0, 0.0), (r, 0.9 * r, r), 1.0, 3.5))
    xyz = torch.stack([x, y, z], -1)
    if not case["down"]:
        return xyz[inside], lab[inside], at, h, body
    blk = (region & inside).view(nz // 2, 2, ny // 2, 2, nx // 2, 2).any(5).any(3).any(1)
    fine = blk.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2) & inside
    mid = xyz.view(nz // 2, 2, ny // 2, 2, nx // 2, 2, 3).mean((1, 3, 5))
    coarse = ~blk & ((mid[..., 0] / (0.98 * h[0])) ** 2 + (mid[..., 1] / (0.98 * h[1])) ** 2 <= 1.0)
    key = torch.arange(x.numel(), device=DEV).view(x.shape)
    k_all = torch.cat([key[fine], key[::2, ::2, ::2][coarse]])
    order = torch.argsort(k_all)
    lab_c = torch.full((int(coarse.sum()),), body, device=DEV, dtype=torch.int32)
    return (torch.cat([xyz[fine], mid[coarse]])[order], torch.cat([lab[fine], lab_c])[order], at, h, body)


def _matrix(case, xyz, at, h, gen):
    """D as voxel-major CSR (row offsets int64, columns int32, FP32 values) on the GPU."""
    B, R, C = case["beams"], case["rows"], case["cols"]
    off = torch.arange(-2, 4, device=DEV)
    p = xyz - torch.tensor(at, device=DEV, dtype=torch.float64)
    ea, eb = 0.98 * h[0], 0.98 * h[1]
    cols, vals, keep = [], [], []
    for b in range(B):
        th = 2.0 * math.pi * b / B
        ex, ey, ux, uy = math.sin(th), -math.cos(th), math.cos(th), math.sin(th)
        qa = (ex / ea) ** 2 + (ey / eb) ** 2
        qb = 2.0 * (xyz[:, 0] * ex / ea ** 2 + xyz[:, 1] * ey / eb ** 2)
        qc = (xyz[:, 0] / ea) ** 2 + (xyz[:, 1] / eb) ** 2 - 1.0
        depth = ((qb + (qb * qb - 4.0 * qa * qc).clamp_min(0.0).sqrt()) / (2.0 * qa)).clamp_min(0.0)
        u, v = p[:, 0] * ux + p[:, 1] * uy, p[:, 2]
        c = torch.floor(u / BEAMLET + 0.5 * C - 0.5).long()[:, None] + off
        r = torch.floor(v / BEAMLET + 0.5 * R - 0.5).long()[:, None] + off
        gu = torch.exp(-(u[:, None] - (c + 0.5 - 0.5 * C) * BEAMLET) ** 2 / (2 * SIGMA ** 2))
        gv = torch.exp(-(v[:, None] - (r + 0.5 - 0.5 * R) * BEAMLET) ** 2 / (2 * SIGMA ** 2))
        val = torch.exp(-MU * depth)[:, None, None] * gv[:, :, None] * gu[:, None, :]
        ok = ((r >= 0) & (r < R))[:, :, None] & ((c >= 0) & (c < C))[:, None, :]
        idx = torch.where(ok, r[:, :, None] * C + c[:, None, :], 0).flatten(1)
        val, ok = val.flatten(1), ok.flatten(1)
        top = torch.zeros(R * C, device=DEV, dtype=torch.float64)
        top.scatter_reduce_(0, idx[ok], val[ok], "amax")
        cols.append((idx + b * R * C).int())
        keep.append(ok & (val >= CUT * top[idx]))
        vals.append(val.float())
    cols, vals, keep = torch.cat(cols, 1), torch.cat(vals, 1), torch.cat(keep, 1)
    ptr = torch.zeros(len(xyz) + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = keep.sum(1).cumsum(0)
    val = vals[keep]
    return ptr, cols[keep], val * (1.0 + 0.01 * (2.0 * torch.rand(len(val), device=DEV, generator=gen) - 1.0))


def _stored(case, col, val):
    """The stored entries' values in FP64: 16-bit storage keeps D_ij / s_i, s_i a beamlet's largest entry."""
    if case["storage"] == "fp32":
        return val.double()
    n = case["beams"] * case["rows"] * case["cols"]
    s = torch.zeros(n, device=DEV).scatter_reduce_(0, col.long(), val, "amax")
    s[s <= 0] = 1.0
    half = torch.float16 if case["storage"] == "fp16" else torch.bfloat16
    return (val / s[col.long()]).to(half).double() * s[col.long()].double()


def _problem(case, seed):
    """Everything about a case's problem, on the GPU."""
    q = types.SimpleNamespace(case=case)
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 3)
    xyz, q.lab, at, h, body = _anatomy(case, seed)
    q.ptr, q.col, q.val = _matrix(case, xyz, at, h, gen)
    q.V, q.N = len(xyz), case["beams"] * case["rows"] * case["cols"]
    q.is_target = np.array([1, 1] + [0] * (body - 1), np.uint8)
    q.under_w = np.array([10.0, 10.0] + [0.0] * (body - 1))
    q.under_t = np.array([1.0, 0.85] + [0.0] * (body - 1))
    q.over_w = np.array([1.0, 1.0] + [1.0] * (body - 2) + [0.1])
    q.over_t = np.array([1.0, 0.85] + [0.6, 0.5, 0.5][: body - 2] + [0.8])
    vol = torch.bincount(q.lab, minlength=body + 1).double().clamp_min(1.0)
    t = lambda a: torch.as_tensor(a, device=DEV, dtype=torch.float64)
    if case["voxelwise"]:   # re-optimisation: the planned dose as both thresholds, under-dose on the target only
        plan = t(q.over_t)[q.lab] * (1.0 + 0.05 * (2.0 * torch.rand(q.V, device=DEV, generator=gen) - 1.0)).double()
        one = torch.ones(q.V, device=DEV, dtype=torch.float64)
        q.terms = (one * t(q.is_target)[q.lab], plan, one, plan)
    else:
        q.terms = tuple(v[q.lab] for v in (t(q.under_w) * t(q.is_target) / vol, t(q.under_t), t(q.over_w) / vol,
                                           t(q.over_t)))
    # a saved pool: the target's outline from each beam in turn, opened by another amount each time
    row = torch.repeat_interleave(torch.arange(q.V, device=DEV), q.ptr[1:] - q.ptr[:-1])
    seen = torch.zeros(q.N, device=DEV, dtype=torch.float64)
    seen.index_add_(0, q.col.long(), q.val.double() * (q.lab[row] < 2).double())
    seen = (seen / seen.max()).cpu().numpy().reshape(case["beams"], case["rows"], case["cols"])
    u = _unit((seed, 2), 8 * case["apertures"] * (1 + case["rows"])).reshape(case["apertures"], 8, 1 + case["rows"])
    q.pool, q.y0 = [], []
    for k in range(case["apertures"]):
        b = k % case["beams"]
        open_ = seen[b] > (0.02 + 0.5 * u[k, 0, 0])
        L = np.where(open_.any(1), open_.argmax(1), 0)
        Rr = np.where(open_.any(1), case["cols"] - open_[:, ::-1].argmax(1), 0)
        cut = np.floor((Rr - L) * 0.5 * u[k, 1, 1:]).astype(int)
        L, Rr = np.where(u[k, 2, 1:] < 0.5, L + cut, L), np.where(u[k, 2, 1:] < 0.5, Rr, Rr - cut)
        q.pool.append((b, np.stack([L, Rr], 1).astype(np.int32)))
        q.y0.append(0.5 + u[k, 3, 0])
    q.x = sum(y * _mask(case, a) for y, a in zip(q.y0, q.pool))     # the pool's fluence, at the prescribed dose
    z = _times(q, q.val.double(), torch.as_tensor(q.x, device=DEV))
    scale = float(z[q.lab == 0].mean())
    q.x = torch.as_tensor(q.x / scale, device=DEV).float()
    q.y0 = np.array(q.y0) / scale
    return q


def _mask(case, aperture):
    m = np.zeros((case["beams"], case["rows"], case["cols"]))
    for r, (lo, hi) in enumerate(aperture[1]):
        m[aperture[0], r, lo:hi] = 1.0
    return m.reshape(-1)


def _times(q, val, x):
    """D x in the type of val."""
    return torch.sparse_csr_tensor(q.ptr, q.col.long(), val, size=(q.V, q.N)) @ x


def _times_t(q, val, p):
    row = torch.repeat_interleave(torch.arange(q.V, device=DEV), q.ptr[1:] - q.ptr[:-1])
    order = torch.argsort(q.col, stable=True)
    ptr = torch.zeros(q.N + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = torch.bincount(q.col, minlength=q.N).cumsum(0)
    return torch.sparse_csr_tensor(ptr, row[order], val[order], size=(q.N, q.V)) @ p


def _gradient(terms, z):
    a, tu, b, to = terms
    under, over = (tu - z).clamp_min(0.0), (z - to).clamp_min(0.0)
    return 2.0 * (b * over - a * under), (a * under ** 2 + b * over ** 2).sum()


def _host_case(q):
    """The arrays a program has read its patient into, in page-locked memory."""
    pin = lambda t: t.cpu().pin_memory().numpy()
    c = q.case
    return types.SimpleNamespace(
        indptr=pin(q.ptr), indices=pin(q.col), data=pin(q.val), voxel_struct=pin(q.lab),
        rows=np.full(c["beams"], c["rows"], np.int32), cols=np.full(c["beams"], c["cols"], np.int32),
        is_target=q.is_target, under_w=q.under_w, under_t=q.under_t, over_w=q.over_w, over_t=q.over_t)


def _options(case):
    return dict(precision=PREC[case["storage"]], mlc_constraint=dao.MLC[case["mlc"]])


# ---- what is measured ---------------------------------------------------------------

def prepare(case, seed):
    torch.cuda.set_device(0)
    kind = case["kind"]
    if kind == "batch":
        plans = [dao.Plan(_host_case(_problem(case, 1000 * seed + i)), **_options(case)) for i in range(case["plans"])]
        return dict(case=case, plans=plans)
    q = _problem(case, seed)
    s = dict(case=case, pool=q.pool, y0=q.y0)
    empty = lambda n: torch.empty(n, device=DEV)
    if kind == "noalloc":
        t = np.stack([q.under_w * q.is_target, q.under_t, q.over_w, q.over_t], 1)
        t[:, [0, 2]] /= np.maximum(torch.bincount(q.lab, minlength=len(t)).cpu().numpy(), 1)[:, None]
        s.update(ptr=q.ptr.int(), col=q.col.int(), val=q.val, x=q.x, lab=q.lab, terms=t, z=empty(q.V), grad=empty(q.V),
                 F=torch.empty(1, device=DEV, dtype=torch.float64))
        return s
    host = _host_case(q)
    if kind == "replan":
        s["host"] = host
        return s
    terms = [v.cpu().numpy() for v in q.terms] if case["voxelwise"] else None
    s["plan"] = dao.Plan(host, voxel_terms=terms, **_options(case))
    if kind == "price":
        s["plan"].import_apertures(q.pool, q.y0)
    elif kind == "dose":
        s.update(x=q.x, z=empty(q.V), grad=empty(q.V))
    elif kind == "prices":
        z = _times(q, q.val.double(), q.x.double())
        s.update(pi=_gradient(q.terms, z)[0].float(), w=empty(q.N))
    return s


def _plan_read(plan, trace):
    z, F = plan.dose()
    aps = plan.apertures()
    return dict(dose=z, objective=np.float32(F), trace=np.asarray(trace, np.float32),
                intensities=plan.intensities().astype(np.float32), beams=np.array([b for b, _ in aps], np.int32),
                leaves=np.stack([lv for _, lv in aps]))


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "plan":
        s["plan"].reset()
        return _plan_read(s["plan"], s["plan"].solve(case["apertures"])[2])
    if kind == "batch":
        for p in s["plans"]:
            p.reset()
        got = dao.batch_solve(s["plans"], case["apertures"], persistent=True)
        return [_plan_read(p, g[2]) for p, g in zip(s["plans"], got)]
    if kind in ("import", "replan"):
        plan = dao.Plan(s["host"], **_options(case)) if kind == "replan" else s["plan"]
        if kind == "import":
            plan.reset()
        F = plan.import_apertures(s["pool"], s["y0"])
        z, Fz = plan.dose()
        y = plan.intensities()
        if kind == "replan":
            plan.close()
        return dict(dose=z, objective=np.float32(Fz), master=np.float32(F), intensities=y.astype(np.float32))
    if kind == "price":
        st, beam, leaves, rc = s["plan"].price()
        return dict(status=int(st), beam=int(beam), leaves=leaves, reduced_cost=np.float32(rc))
    if kind == "dose":
        F = s["plan"].k_dose(s["x"], s["z"], s["grad"])
        return dict(dose=s["z"], gradient=s["grad"], objective=np.float32(F))
    if kind == "prices":
        s["plan"].k_beamlet_prices(s["pi"], s["w"])
        return dict(prices=s["w"])
    dao.dose_objective_noalloc(s["ptr"], s["col"], s["val"], s["x"], s["lab"], s["terms"], s["z"], s["grad"], s["F"])
    return dict(dose=s["z"], gradient=s["grad"], objective=s["F"].float())


# ---- 64-bit values -------------------------------------------------------------------

def _master64(S, terms, y):
    """min F(S y), y >= 0, by projected Newton from y."""
    def at(v):
        z = S @ v
        pi, F = _gradient(terms, z)
        return z, F, S.T @ pi
    z, F, g = at(y)
    stop = 1e-13 * float(g.abs().max()) + 1e-300
    for _ in range(200):
        if float((y - (y - g).clamp_min(0.0)).abs().max()) <= stop:
            break
        h = 2.0 * (terms[0] * (z < terms[1]) + terms[2] * (z > terms[3]))
        free = ~((y <= 1e-12) & (g > 0))
        d = torch.where(free, torch.zeros_like(g), -g)
        Sf = S[:, free]
        H = Sf.T @ (h[:, None] * Sf)
        H += 1e-13 * H.diagonal().max() * torch.eye(len(H), device=DEV, dtype=H.dtype)
        d[free] = -torch.linalg.solve(H, g[free])
        a = 1.0
        while a > 1e-12:
            yt = (y + a * d).clamp_min(0.0)
            zt, Ft, gt = at(yt)
            if Ft <= F + 1e-4 * (g @ (yt - y)):
                break
            a *= 0.5
        else:
            break
        y, z, F, g = yt, zt, Ft, gt
    return y, z, F


def _price64(case, w):
    """(beam, leaves, value) of the aperture with the smallest reduced cost for beamlet prices w."""
    best = None
    for b, wb in enumerate(w.reshape(case["beams"], case["rows"], case["cols"])):
        P = np.concatenate([np.zeros((case["rows"], 1)), np.cumsum(wb, 1)], 1)
        if case["mlc"] == "consecutive":
            m = np.maximum.accumulate(P[:, :-1], 1)
            hi = (P[:, 1:] - m).argmin(1)
            lo = np.array([P[r, : hi[r] + 1].argmax() for r in range(case["rows"])])
            v = np.minimum((P[:, 1:] - m).min(1), 0.0)
            lr, total = np.where((v < 0)[:, None], np.stack([lo, hi + 1], 1), 0), float(v.sum())
        else:   # leaves of adjacent rows may not cross
            s = [(i, j) for i in range(case["cols"] + 1) for j in range(i, case["cols"] + 1)]
            lo, hi = np.array([i for i, _ in s]), np.array([j for _, j in s])
            fits = (lo[None, :] <= hi[:, None]) & (lo[:, None] <= hi[None, :])
            f = P[0, hi] - P[0, lo]
            for r in range(1, case["rows"]):
                f = P[r, hi] - P[r, lo] + np.where(fits, f[None, :], np.inf).min(1)
            lr, total = None, min(float(f.min()), 0.0)
        if best is None or total < best[2]:
            best = (b, lr, total)
    return best


def _column64(q, val, aperture):
    return _times(q, val, torch.as_tensor(_mask(q.case, aperture), device=DEV))


def _plan64(q):
    val = _stored(q.case, q.col, q.val)
    S = torch.zeros(q.V, 0, device=DEV, dtype=torch.float64)
    y, z, trace = S.new_zeros(0), S.new_zeros(q.V), []
    for _ in range(q.case["apertures"]):
        w = _times_t(q, val, _gradient(q.terms, z)[0]).cpu().numpy()
        b, lr, _ = _price64(q.case, w)
        S = torch.cat([S, _column64(q, val, (b, lr))[:, None]], 1)
        y, z, F = _master64(S, q.terms, torch.cat([y, y.new_zeros(1)]))
        trace.append(float(F))
    return dict(dose=z, objective=trace[-1], trace=np.array(trace), intensities=None, beams=None, leaves=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_plan64(_problem(case, 1000 * seed + i)) for i in range(case["plans"])]
    q = _problem(case, seed)
    if kind == "plan":
        return _plan64(q)
    val = _stored(case, q.col, q.val)
    if kind in ("import", "replan", "price"):
        S = torch.stack([_column64(q, val, a) for a in q.pool], 1)
        _, z, F = _master64(S, q.terms, torch.as_tensor(q.y0, device=DEV))
        if kind == "price":
            w = _times_t(q, val, _gradient(q.terms, z)[0]).cpu().numpy()
            return dict(status=None, beam=None, leaves=None, reduced_cost=_price64(case, w)[2])
        return dict(dose=z, objective=float(F), master=float(F), intensities=None)
    z = _times(q, val, q.x.double())
    pi, F = _gradient(q.terms, z)
    if kind == "prices":
        z = _times(q, q.val.double(), q.x.double())
        return dict(prices=_times_t(q, val, _gradient(q.terms, z)[0].float().double()))
    return dict(dose=z, gradient=pi, objective=float(F))


# ---- what a pass cannot do without -----------------------------------------------------

@functools.lru_cache(maxsize=None)
def _sizes(nx, ny, nz, down, beams, rows, cols):
    c = dict(nx=nx, ny=ny, nz=nz, down=down, beams=beams, rows=rows, cols=cols)
    xyz, _, at, h, _ = _anatomy(c, 0)
    return len(xyz), int(_matrix(c, xyz, at, h, torch.Generator(device=DEV).manual_seed(0))[0][-1])


def work(case):
    V, nnz = _sizes(*(case[k] for k in ("nx", "ny", "nz", "down", "beams", "rows", "cols")))
    N, B, K, vb, kind = case["beams"] * case["rows"] * case["cols"], case["beams"], case["apertures"], \
        VALUE_BYTES[case["storage"]], case["kind"]
    idx = 4 if case["storage"] == "fp32" else 2           # a beamlet index
    d = (idx + vb) * nnz + 4 * V                          # D by voxels
    dt = (4 + vb) * nnz + 4 * N                           # D by beamlets
    column = (2 + vb) * nnz / B + 8 * V                   # one beam's part of D, and the column
    crit = 32 * V if case["voxelwise"] else V             # the criteria of every voxel
    if kind == "dose":
        return dict(bytes=d + 4 * N + 8 * V + crit, flops=2 * nnz + 8 * V)
    if kind == "noalloc":
        return dict(bytes=8 * nnz + 8 * V + 4 * N + 8 * V, flops=2 * nnz + 8 * V)
    if kind == "prices":
        return dict(bytes=dt + 4 * V + 4 * N, flops=2 * nnz)
    if kind == "price":
        return dict(bytes=dt + 4 * V + 16 * N, flops=2 * nnz + 4 * N)
    # a master solve reads the pool's columns once and writes the dose and the dual
    master = lambda k: 4.0 * V * k + crit + 8 * V
    mflops = lambda k: 2.0 * V * k * 3
    if kind in ("import", "replan"):
        b, f = K * column + master(K) + d + 8 * V, K * 2.0 * nnz / B + mflops(K) + 2 * nnz
        return dict(bytes=b + (8 * nnz + 12 * V + d + dt + (2 + vb) * nnz if kind == "replan" else 0), flops=f)
    b = sum(dt + 4 * V + 4 * N + column + master(k) for k in range(1, K + 1)) + d + 8 * V
    f = sum(2.0 * nnz + 2.0 * nnz / B + mflops(k) for k in range(1, K + 1)) + 2 * nnz
    return dict(bytes=b * case["plans"], flops=f * case["plans"])
