"""The work a user of the level solver has it do, as timed cases.

A case is a plain dict.  ``kind`` says which public call it goes through:

  solve   one level: ``Level.build`` (the step's K, E^n and wall values), then
          ``Level.solve``
  batch   many ragged levels: ``Batch.build_operators``, then ``Batch.solve``
  amr     one coarse step of a two-level heat hierarchy
  fld     one coarse step of the four-level radiation-matter hierarchy
  serve   a burst of requests through the serving loop

Every solve stops on the certificate ||b - A x|| <= 5e-11 ||x||, the rule of
the repository's configurations, which bounds the relative error of x itself
(the residual-relative rule does not).  Sizes, time steps and fields follow the
repository's five workload configurations: cells K = exp(N(0, 1)), E uniform in
[0.5, 1.5], walls zero-flux, Dirichlet or Robin, time steps in explicit CFL
units dx^2 / 2.
"""
import math
import types

import numpy as np
import torch

from paper_1401_1112_gb300 import ats

TOL = 5e-11
DIRICHLET, NEUMANN, ROBIN = 0, 1, 2


def listed():
    return [
        # the smallest level a hierarchy or a batch holds, solved alone: launches and host work count
        {"name": "solve_8cube_mixed", "kind": "solve", "nx": 4, "ny": 4, "nz": 4, "cfl": 10.0, "prec": "mixed",
         "walls": "zero", "field": "random", "mem": "device"},
        # configuration 1: 32^3 Gaussian, zero-flux walls, ten explicit steps, the default (FP64) precision
        {"name": "solve_32cube_fp64", "kind": "solve", "nx": 16, "ny": 16, "nz": 16, "cfl": 10.0, "prec": "fp64",
         "walls": "zero", "field": "gauss", "mem": "device"},
        # a ragged mid-size level from pageable numpy arrays, as a host code calls the library
        {"name": "solve_ragged_host_mixed", "kind": "solve", "nx": 21, "ny": 17, "nz": 19, "cfl": 30.0,
         "prec": "mixed", "walls": "mixed", "field": "random", "mem": "host"},
        # a level of the two-level hierarchy's size alone, FP64
        {"name": "solve_64cube_fp64", "kind": "solve", "nx": 31, "ny": 33, "nz": 32, "cfl": 10.0, "prec": "fp64",
         "walls": "mixed", "field": "random", "mem": "device"},
        # the same size in mixed precision with a stiff step
        {"name": "solve_64cube_mixed", "kind": "solve", "nx": 32, "ny": 32, "nz": 32, "cfl": 30.0, "prec": "mixed",
         "walls": "mixed", "field": "random", "mem": "device"},
        # a large served / base level
        {"name": "solve_160cube_mixed", "kind": "solve", "nx": 80, "ny": 79, "nz": 81, "cfl": 30.0, "prec": "mixed",
         "walls": "mixed", "field": "random", "mem": "device"},
        # configuration 4: 512 ragged levels of 8^3 .. 64^3 cells in one batch, every level on the resident solver as
        # the repository's benchmark asks for
        {"name": "batch_512_mixed", "kind": "batch", "n": 512, "lo": 64, "hi": 32768, "cfl_lo": 1e-3, "cfl_hi": 1e2,
         "prec": "mixed", "cn": False, "mem": "device", "res_max": 32768},
        # the same mix, fewer levels, Crank-Nicolson, from and to pinned host memory
        {"name": "batch_96_cn_host", "kind": "batch", "n": 96, "lo": 64, "hi": 16384, "cfl_lo": 1e-3, "cfl_hi": 1e2,
         "prec": "mixed", "cn": True, "mem": "host", "res_max": 0},
        # many small levels in FP64 (the finest levels of a hierarchy, the default precision)
        {"name": "batch_128_small_fp64", "kind": "batch", "n": 128, "lo": 64, "hi": 2048, "cfl_lo": 1e-2,
         "cfl_hi": 1e2, "prec": "fp64", "cn": False, "mem": "device", "res_max": 0},
        # configuration 2: base 64^3 plus a refined central eighth, fine level first, the step replayed as one graph
        {"name": "amr_two_level_64cube", "kind": "amr", "n0": 64, "cfl": 10.0, "prec": "mixed", "graph": 3},
        # configuration 3 at a 64^3 base: four levels that a remeshing code builds anew, steps enqueued without a graph
        {"name": "fld_four_level_64cube", "kind": "fld", "n0": 64, "levels": 4, "cfl": 30.0, "prec": "mixed",
         "graph": 2},
        # configuration 5: a burst of requests, 16^3 .. 64^3 cells, all three wall kinds
        {"name": "serve_24_mixed", "kind": "serve", "n": 24, "lo": 512, "hi": 32768, "cfl_lo": 1e-3, "cfl_hi": 1e2,
         "prec": "mixed"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "batch", "amr", "fld", "serve"])
    prec = "fp64" if rng.random() < 0.3 else "mixed"
    if kind == "solve":
        n = _log(rng, 64, 65536 if prec == "fp64" else 400000)
        a = max(1, round(n ** (1 / 3) * rng.uniform(0.7, 1.4)))
        b = max(1, round(math.sqrt(n / a) * rng.uniform(0.8, 1.25)))
        return {"kind": kind, "nx": a, "ny": b, "nz": max(1, round(n / (a * b))), "cfl": round(_log(rng, 1e-2, 50), 4),
                "prec": prec, "walls": rng.choice(["zero", "mixed"]), "field": rng.choice(["gauss", "random"]),
                "mem": "host" if n < 20000 and rng.random() < 0.3 else "device"}
    if kind == "batch":
        hi = 2048 if prec == "fp64" else rng.choice([1024, 8192, 32768])
        return {"kind": kind, "n": int(_log(rng, 4, 160)), "lo": 64, "hi": hi, "cfl_lo": 1e-3, "cfl_hi": 1e2,
                "prec": prec, "cn": rng.random() < 0.3, "mem": rng.choice(["device", "host"]),
                "res_max": 0 if prec == "fp64" else rng.choice([0, 32768])}
    if kind == "amr":
        return {"kind": kind, "n0": 4 * rng.randint(5, 15), "cfl": round(rng.uniform(2, 15), 3), "prec": prec,
                "graph": rng.choice([2, 3])}
    if kind == "fld":
        return {"kind": kind, "n0": 2 * rng.randint(16, 30), "levels": rng.randint(2, 4),
                "cfl": round(rng.uniform(5, 30), 3), "prec": "mixed", "graph": 2}
    return {"kind": kind, "n": rng.randint(2, 24), "lo": 64, "hi": rng.choice([2048, 16384]), "cfl_lo": 1e-3,
            "cfl_hi": 1e2, "prec": "mixed"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _morton(xyz):
    """Order of the octs along a Morton curve."""
    v = xyz.astype(np.int64) - xyz.min(axis=0)
    key = np.zeros(len(v), np.int64)
    for bit in range(int(v.max()).bit_length() if len(v) else 0):
        for a in range(3):
            key |= ((v[:, a] >> bit) & 1) << (3 * bit + a)
    return np.argsort(key, kind="stable")


def _cells(xyz):
    c = np.arange(8)
    return (2 * xyz.astype(np.int64)[:, None, :] + np.stack([c & 1, c >> 1 & 1, c >> 2], 1)[None]).reshape(-1, 3)


def _level(xyz, dx, leaf=None, faces=None):
    """A level description as the library takes it; faces: (cell, dir, kind, alpha) of the wall descriptors."""
    cell, dr, kind, alpha = faces if faces is not None else (np.zeros(0),) * 4
    return types.SimpleNamespace(
        oct_xyz=np.ascontiguousarray(xyz, dtype=np.int32), leaf=leaf, dx=float(dx), n_cell=8 * len(xyz),
        face_cell=np.ascontiguousarray(cell, np.int32), face_dir=np.ascontiguousarray(dr, np.int8),
        face_kind=np.ascontiguousarray(kind, np.int8), face_rel=np.zeros(len(cell), np.int8),
        face_alpha=np.ascontiguousarray(alpha, np.float64))


def _box(nx, ny, nz, walls):
    """A full box of octs; walls: per side None (zero flux) or (kind, alpha, E, F).  Returns the level and the
    descriptors' E and F."""
    xyz = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1).reshape(-1, 3)
    xyz = xyz[_morton(xyz)].astype(np.int32)
    cell, side = [], []
    for d, w in enumerate(walls):
        if w is None:
            continue
        a, s = d >> 1, d & 1
        on = np.nonzero(xyz[:, a] == ((nx, ny, nz)[a] - 1 if s else 0))[0]
        c = np.array([c for c in range(8) if (c >> a & 1) == s])
        cell.append((8 * on[:, None] + c[None]).reshape(-1))
        side.append(np.full(len(cell[-1]), d))
    dx = 1.0 / (2 * max(nx, ny, nz))
    if not cell:
        return _level(xyz, dx), np.zeros(0), np.zeros(0)
    cell, side = np.concatenate(cell), np.concatenate(side)
    order = np.lexsort((side, cell))
    cell, side = cell[order], side[order]
    at = lambda k: np.array([w[k] if w else 0 for w in walls], np.float64)[side]  # noqa: E731
    return _level(xyz, dx, faces=(cell, side, at(0), at(1))), at(2), at(3)


def _walls(rng, how):
    """zero: none; dirichlet: each side zero-flux or Dirichlet; mixed: Dirichlet, Neumann or Robin with a flux."""
    out = []
    for _ in range(6):
        e, f, al = float(rng.uniform(0, 2)), float(rng.uniform(-0.05, 0.05)), float(rng.uniform(0, 1))
        if how == "zero" or (how == "dirichlet" and rng.uniform() < 0.5):
            out.append(None)
        elif how == "dirichlet":
            out.append((DIRICHLET, 1.0, e, 0.0))
        else:
            k = int(rng.integers(0, 3))
            out.append((k, (1.0, 0.0, al)[k], e, f))
    return out


def _near_cubic(o):
    a = max(1, round(o ** (1 / 3)))
    b = max(1, round(math.sqrt(o / a)))
    return a, b, max(1, round(o / (a * b)))


def _gpu_random(seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed)
    K = torch.exp(torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    return K, torch.rand(n, generator=g, device="cuda", dtype=torch.float64) + 0.5


def _gaussian(lv, sigma, floor):
    xyz = (_cells(lv.oct_xyz) + 0.5) * lv.dx - 0.5
    return np.exp(-(xyz ** 2).sum(1) / (2 * sigma * sigma)) + floor


def _boxes(case, seed):
    """The levels of a solve, batch or serve case: (level, dt, wall E, wall F) each, and all cells' K and E^n."""
    rng = np.random.default_rng(seed)
    out = []
    if case["kind"] == "solve":
        lv, fE, fF = _box(case["nx"], case["ny"], case["nz"], _walls(rng, case["walls"]))
        out.append((lv, case["cfl"] * lv.dx ** 2 / 2, fE, fF))
    else:
        how = "mixed" if case["kind"] == "serve" else "dirichlet"
        # sizes and steps belong to the case: the whole range of each, one of each stratum, in random order
        n, fixed = case["n"], np.random.default_rng(case["n"])
        size = (np.arange(n) + fixed.uniform(0, 1, n)) / n
        step = (fixed.permutation(n) + fixed.uniform(0, 1, n)) / n
        for k in fixed.permutation(n):
            o = case["lo"] * (case["hi"] / case["lo"]) ** size[k]
            lv, fE, fF = _box(*_near_cubic(round(o)), _walls(rng, how))
            out.append((lv, case["cfl_lo"] * (case["cfl_hi"] / case["cfl_lo"]) ** step[k] * lv.dx ** 2 / 2, fE, fF))
    K, E = _gpu_random(seed, sum(b[0].n_cell for b in out))
    if case.get("field") == "gauss":
        K = torch.ones_like(K)
        E = torch.from_numpy(_gaussian(out[0][0], 0.05, 1e-3)).cuda() * (1 + 1e-3 * E)
    return out, K, E


def _hierarchy(case, seed):
    """Levels, per-level E and (heat) K or (fld) rho on the GPU, the coarse step and k0."""
    n0, rng = case["n0"], np.random.default_rng(seed)
    dx0 = 1.0 / n0
    g = np.stack(np.meshgrid(*[np.arange(n0 // 2)] * 3, indexing="ij"), -1).reshape(-1, 3)
    octs = g[_morton(g)]
    key = lambda c: (c[:, 0] << 40) | (c[:, 1] << 20) | c[:, 2]  # noqa: E731
    if case["kind"] == "fld":
        # the mesh belongs to the case: it follows one log-normal density; the seed varies the values on it
        field = np.exp(1.5 * np.random.default_rng(n0).standard_normal((n0, n0, n0)))
        field /= field.mean()
    rho_mean = None
    levels, rhos = [], []
    n_levels = 2 if case["kind"] == "amr" else case["levels"]
    for l in range(n_levels):
        dx, cells = dx0 / 2 ** l, _cells(octs)
        want = np.zeros(len(cells), bool)
        if case["kind"] == "amr":
            if l == 0:
                want = np.all((cells >= n0 // 4) & (cells < 3 * n0 // 4), axis=1)
        else:
            rho = _density(field, (cells + 0.5) * dx - 0.5)
            rhos.append(rho)
            rho_mean = rho.mean() if l == 0 else rho_mean
            if l + 1 < n_levels:
                want = rho > 4.0 ** (l + 1) * rho_mean
                have, nl = key(cells), n0 << l
                for a in range(3):  # 2:1 balance: every neighbour inside the domain exists at this level
                    for s in (-1, 1):
                        q = cells.copy()
                        q[:, a] += s
                        inside = (q[:, a] >= 0) & (q[:, a] < nl)
                        want[inside] &= np.isin(key(q[inside]), have)
        leaf = np.zeros(len(octs), np.uint8)
        for c in range(8):
            leaf |= (~want.reshape(-1, 8)[:, c]).astype(np.uint8) << np.uint8(c)
        levels.append(_level(octs, dx, leaf=leaf))
        octs = cells[want]
        if not len(octs):
            break
        octs = octs[_morton(octs)]
    gpu = lambda v: torch.from_numpy(np.ascontiguousarray(v, np.float64)).cuda()  # noqa: E731
    if case["kind"] == "amr":
        # Gaussian pulse, K = 1 up to a seeded one per cent
        E = [gpu(_gaussian(lv, 0.05, 1e-3)) for lv in levels]
        X = [gpu(1 + 0.01 * rng.standard_normal(lv.n_cell)) for lv in levels]
        return levels, E, X, case["cfl"] * dx0 ** 2 / 2, None
    E = [gpu(1 + 10 * _gaussian(lv, 0.05, 0.0)) for lv in levels]
    k0 = 1.0 / (np.median(rhos[0] ** 2) * dx0)  # median base-cell optical depth 1: K about dx0 / 3 there
    rhos = [r * np.exp(0.1 * rng.standard_normal(len(r))) for r in rhos]
    return levels, E, [gpu(r) for r in rhos], case["cfl"] * dx0 ** 2 / (2 * dx0 / 3), float(k0)


def _density(field, pts):
    """Trilinear interpolation of the base field times a central core 1 / (1 + (r / 0.05)^2)."""
    n = field.shape[0]
    u = (pts + 0.5) * n - 0.5
    i0 = np.clip(np.floor(u).astype(np.int64), 0, n - 1)
    i1, f, out = np.clip(i0 + 1, 0, n - 1), np.clip(u - i0, 0, 1), 0.0
    for c in range(8):
        b = np.array([c & 1, c >> 1 & 1, c >> 2], bool)
        i, w = np.where(b, i1, i0), np.where(b, f, 1 - f).prod(1)
        out = out + w * field[i[:, 0], i[:, 1], i[:, 2]]
    return out / (1 + (pts ** 2).sum(1) / 0.0025)


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

class _State:
    """Handles that a user's program keeps, closed with the state, the context last."""

    def __init__(self, case):
        self.case, self.handles = case, []

    def own(self, handle):
        self.handles.append(handle)
        return handle

    def __del__(self):
        for h in reversed(self.handles):
            h.close()


def prepare(case, seed):
    st = _State(case)
    prec = ats.ATS_PREC_MIXED if case["prec"] == "mixed" else ats.ATS_PREC_FP64
    st.opts = dict(tol=TOL, stop_rule=ats.ATS_STOP_CERTIFIED, precision=prec, x0=ats.ATS_X0_E_OLD)
    if case["kind"] in ("amr", "fld"):
        ctx = st.own(ats.Context(0))
        st.levels, st.E, st.X, st.dt, st.k0 = _hierarchy(case, seed)
        order = ats.ATS_ORDER_FINE_FIRST
        st.h = st.own(ats.Hierarchy(ctx, st.levels, order=order))
        st.T = [torch.ones_like(e) for e in st.E]
        st.one = [torch.ones_like(e) for e in st.E]
        st.out = [torch.empty_like(e) for e in st.E]
        st.out_T = [torch.empty_like(e) for e in st.E] if case["kind"] == "fld" else []
        st.opts.update(use_graph=case["graph"], x0=ats.ATS_X0_GIVEN)
        torch.cuda.synchronize()
        return st
    boxes, K, E = _boxes(case, seed)
    off = np.cumsum([0] + [b[0].n_cell for b in boxes])
    if case["kind"] == "serve":
        K, E = K.cpu().numpy(), E.cpu().numpy()
        del st.opts["x0"]
        st.server = st.own(ats.Server(precision=prec))
        # a first small request: the scheduler thread has recorded its graph once it is answered
        lv = _box(1, 1, 1, [None] * 6)[0]
        one = types.SimpleNamespace(dt=1e-3, K=np.ones(8), E=np.ones(8), face_K=None, face_E=None, face_F=None, s=None,
                                    src=None)
        st.server.wait(st.server.submit(lv, one), 8)
        st.reqs = [(lv, types.SimpleNamespace(dt=dt, K=K[i:j], E=E[i:j], face_K=None, face_E=fE if len(fE) else None,
                                              face_F=fF if len(fF) else None, s=None, src=None))
                   for (lv, dt, fE, fF), i, j in zip(boxes, off[:-1], off[1:])]
        torch.cuda.synchronize()
        return st
    host = case["mem"] == "host"
    if host:
        pin = case["kind"] == "batch"  # a program that pipelines batches pins its buffers
        move = lambda t: (t.cpu().pin_memory() if pin else t.cpu()).numpy()  # noqa: E731
    else:
        move = lambda t: t.cuda()  # noqa: E731
    st.x = torch.empty(int(off[-1]), dtype=torch.float64, device="cpu" if host else "cuda",
                       pin_memory=host and case["kind"] == "batch")
    x = st.x.numpy() if host else st.x
    # one buffer per kind of array, the levels' slices after one another
    K, E = move(K), move(E)
    foff = np.cumsum([0] + [len(b[2]) for b in boxes])
    fE, fF = (move(torch.from_numpy(np.concatenate([b[k] for b in boxes]))) for k in (2, 3))
    ctx = st.own(ats.Context(0))
    st.levels = [st.own(ats.Level(ctx, b[0])) for b in boxes]
    st.xs = [x[i:j] for i, j in zip(off[:-1], off[1:])]
    st.coefs = []
    for k, (lv, dt, wE, _) in enumerate(boxes):
        c = dict(dt=dt, K=K[off[k]:off[k + 1]], E_old=E[off[k]:off[k + 1]])
        if len(wE):
            c.update(face_E=fE[foff[k]:foff[k + 1]], face_F=fF[foff[k]:foff[k + 1]])
        if case.get("cn"):
            c["integrator"] = ats.ATS_INTEGRATOR_CRANK_NICOLSON
        st.coefs.append(c)
    torch.cuda.synchronize()
    if case["kind"] == "batch":
        for lv, c in zip(st.levels, st.coefs):  # a batch is planned over built levels
            lv.build(c["dt"], **{k: v for k, v in c.items() if k != "dt"})
        st.opts.update(mem=ats.ATS_MEM_HOST if host else ats.ATS_MEM_DEVICE, use_graph=2,
                       res_max_octs=case["res_max"])
        st.batch = st.own(ats.Batch(ctx, st.levels, **st.opts))
        st.prepared = st.batch.prepare_coefs(st.coefs)
        torch.cuda.synchronize()
    return st


def _ok(code):
    if code < 0:
        raise RuntimeError(ats.ats_status_string(code))


def run(st):
    kind = st.case["kind"]
    if kind == "solve":
        c = st.coefs[0]
        st.levels[0].build(c["dt"], c["K"], c["E_old"], face_E=c.get("face_E"), face_F=c.get("face_F"))
        _ok(st.levels[0].solve(st.xs[0], **st.opts)[0])
        return st.x
    if kind == "batch":
        st.batch.build_operators(st.prepared)
        _ok(st.batch.solve(st.xs)[0])
        return st.x
    if kind == "serve":
        tickets = [st.server.submit(lv, step, tol=TOL, stop_rule=ats.ATS_STOP_CERTIFIED) for lv, step in st.reqs]
        out = [st.server.wait(t, lv.n_cell) for t, (lv, _) in zip(tickets, st.reqs)]
        for code, _, _ in out:
            _ok(code)
        return [x for _, x, _ in out]
    for l, e in enumerate(st.E):
        st.h.set_state(l, e, st.X[l] if kind == "amr" else st.one[l])
        if kind == "fld":
            st.h.set_fld(l, st.X[l], st.T[l], st.k0)
    _ok(st.h.advance(0, st.dt, **st.opts)[0])
    for l in range(len(st.E)):
        ats.ats_hierarchy_get_state(st.h.handle, l, st.out[l])
        if kind == "fld":
            ats.ats_hierarchy_get_temperature(st.h.handle, l, st.out_T[l])
    return st.out + st.out_T


def work(case):
    """Inputs and the result once (K, E^n, x in FP64), and the floating-point operations of an estimated number of CG
    iterations: 12 sqrt(1 + 8 h) per solve, h = dt / (2 dx^2), about 31 per cell and iteration (stencil 19, vector
    updates 8, sums 4)."""
    its = lambda cfl: 12 * math.sqrt(1 + 2 * cfl)  # noqa: E731
    if case["kind"] == "solve":
        n = 8 * case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 24 * n, "flops": 31 * n * its(case["cfl"])}
    if case["kind"] in ("batch", "serve"):
        n = 8 * case["n"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        q = (np.arange(64) + 0.5) / 64
        mean = float(np.mean([its(case["cfl_lo"] * (case["cfl_hi"] / case["cfl_lo"]) ** v) for v in q]))
        return {"bytes": 24 * n, "flops": 31 * n * mean}
    # per level: the base once, finer levels 2^l times; refined cells a fixed share of the base
    n = case["n0"] ** 3
    cells = n + 2 * n if case["kind"] == "amr" else 1.8 * n
    return {"bytes": 24 * cells, "flops": 31 * cells * its(case["cfl"])}


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------

class _Grid:
    """Cells (grid id, x, y, z) with their same-grid neighbours, by sorted keys."""

    def __init__(self, sid, xyz):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        c = torch.from_numpy(np.column_stack([sid, xyz])).to(self.dev) + 2
        key = lambda c: (c[:, 0] << 45) | (c[:, 1] << 30) | (c[:, 2] << 15) | c[:, 3]  # noqa: E731
        self.sorted, order = torch.sort(key(c))
        self.nb = torch.empty(6, len(c), dtype=torch.int64, device=self.dev)
        for d in range(6):
            q = c.clone()
            q[:, 1 + (d >> 1)] += 2 * (d & 1) - 1
            k = key(q)
            at = torch.searchsorted(self.sorted, k).clamp(max=len(c) - 1)
            self.nb[d] = torch.where(self.sorted[at] == k, order[at], -1)


def _cg(nb, C, diag, b, x, leaf):
    """Jacobi-CG for diag x - sum_d C[d] x[nb[d]] = b on the leaf cells, to a residual of 1e-15 |x|."""
    nb = nb.clamp(min=0)

    def mul(v):
        y = diag * v
        for d in range(6):
            y -= C[d] * v[nb[d]]
        return torch.where(leaf, y, 0.0)

    keep, x = x, torch.where(leaf, x, 0.0)
    for _ in range(2):  # restarted from the true residual
        r = torch.where(leaf, b, 0.0) - mul(x)
        z = r / diag
        p, rz = z.clone(), r @ z
        for it in range(4000):
            if it % 8 == 0 and float(r.norm()) <= 1e-15 * float(x.norm()):
                break
            q = mul(p)
            alpha = rz / (p @ q)
            x, r = x + alpha * p, r - alpha * q
            z = r / diag
            rz, old = r @ z, rz
            p = z + (rz / old) * p
    return torch.where(leaf, x, keep)


def exact(case, seed):
    if case["kind"] in ("amr", "fld"):
        return _exact_hierarchy(case, seed)
    boxes, K, E = _boxes(case, seed)
    off = np.cumsum([0] + [b[0].n_cell for b in boxes])
    grid = _Grid(np.repeat(np.arange(len(boxes)), np.diff(off)), np.concatenate([_cells(b[0].oct_xyz) for b in boxes]))
    K, E = K.to(grid.dev), E.to(grid.dev)
    put = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(grid.dev)  # noqa: E731
    half = 0.5 if case.get("cn") else 1.0  # Crank-Nicolson: 2 x' - E^n, x' the half step's backward-Euler root
    h = put(np.repeat([half * b[1] / (2 * b[0].dx ** 2) for b in boxes], np.diff(off)))
    C = torch.where(grid.nb >= 0, h * (K + K[grid.nb.clamp(min=0)]), 0.0)
    diag, rhs = 1 + C.sum(0), E.clone()
    cell = put(np.concatenate([b[0].face_cell.astype(np.int64) + o for b, o in zip(boxes, off)]))
    if len(cell):
        al = put(np.concatenate([b[0].face_alpha for b in boxes]))  # 1 Dirichlet, 0 Neumann
        fE, fF = (put(np.concatenate([b[k] for b in boxes])) for k in (2, 3))
        Cf = al * 2 * h[cell] * K[cell]
        diag.index_add_(0, cell, Cf)
        rhs.index_add_(0, cell, Cf * fE + (1 - al) * half * fF)
    x = _cg(grid.nb, C, diag, rhs, E, torch.ones_like(E, dtype=torch.bool))
    x = 2 * x - E if case.get("cn") else x
    if case["kind"] == "serve":
        return [x[i:j] for i, j in zip(off[:-1], off[1:])]
    return x


def _exact_hierarchy(case, seed):
    """Fine levels first, two half steps each, the coarse neighbour held; a refined cell is its children's mean."""
    levels, E, X, dt0, k0 = _hierarchy(case, seed)
    fld, dev, n = case["kind"] == "fld", E[0].device, len(levels)
    K = [torch.ones_like(e) for e in E] if fld else [k.clone() for k in X]
    E, T = [e.clone() for e in E], [torch.ones_like(e) for e in E]
    cells = [_cells(lv.oct_xyz) for lv in levels]
    leaf = [torch.from_numpy((lv.leaf[:, None] >> np.arange(8) & 1).reshape(-1).astype(bool)).to(dev) for lv in levels]
    nb = [_Grid(np.zeros(len(c), np.int64), c).nb.to(dev) for c in cells]
    pack = lambda c: torch.from_numpy((c[:, 0] << 40) | (c[:, 1] << 20) | c[:, 2]).to(dev)  # noqa: E731
    order = [torch.sort(pack(c)) for c in cells]

    def find(l, c):
        k = pack(c)
        at = torch.searchsorted(order[l].values, k).clamp(max=len(order[l].values) - 1)
        return torch.where(order[l].values[at] == k, order[l].indices[at], -1)

    up = [None] + [find(l - 1, levels[l].oct_xyz.astype(np.int64)) for l in range(1, n)]
    beyond = [None]  # per direction the coarser cell across a face that has no cell of this level, or -1
    for l in range(1, n):
        rows = []
        for d in range(6):
            q = cells[l].copy()
            q[:, d >> 1] += 2 * (d & 1) - 1
            inside = torch.from_numpy(np.all((q >= 0) & (q < case["n0"] << l), axis=1)).to(dev)
            rows.append(torch.where(inside, find(l - 1, q >> 1), -1))
        beyond.append(torch.stack(rows))

    def model(l, dt):
        kr = k0 * X[l] ** 2 / T[l]
        g2 = 0.0
        for a in range(3):
            lo, hi = nb[l][2 * a], nb[l][2 * a + 1]
            d = torch.where(hi >= 0, E[l][hi.clamp(min=0)], E[l]) - torch.where(lo >= 0, E[l][lo.clamp(min=0)], E[l])
            g2 = g2 + (d / (levels[l].dx * ((hi >= 0).double() + (lo >= 0).double()).clamp(min=1))) ** 2
        R = g2.sqrt() / (kr * E[l])
        K[l] = torch.where(leaf[l], (2 + R) / (6 + 3 * R + R * R) / kr, K[l])
        sigma, mu = dt * kr, 4 * T[l] ** 3 / X[l]
        return sigma, mu

    for l in range(n if fld else 0):
        model(l, 1.0)  # the coefficients of the initial state (dt does not enter them)

    def advance(l, dt):
        if l + 1 < n:
            advance(l + 1, dt / 2)
            advance(l + 1, dt / 2)
            for V in (E, K):
                V[l][up[l + 1]] = V[l + 1].reshape(-1, 8).mean(1)
        shift = src = 0.0
        if fld:
            sigma, mu = model(l, dt)
            shift = sigma / (1 + sigma * mu)
            src = shift * T[l] ** 4
        h = dt / (2 * levels[l].dx ** 2)
        j = nb[l].clamp(min=0)
        C = torch.where(nb[l] >= 0, h * (K[l] + K[l][j]), 0.0)
        inner = leaf[l][j] & (nb[l] >= 0)
        rhs = E[l] + src + torch.where(inner, 0.0, C * E[l][j]).sum(0)  # a refined neighbour: its mean, held
        diag = 1 + shift + C.sum(0)
        if l:
            jc = beyond[l].clamp(min=0)
            Cc = torch.where((nb[l] < 0) & (beyond[l] >= 0), 2 / 3 * h * (K[l] + K[l - 1][jc]), 0.0)
            rhs, diag = rhs + (Cc * E[l - 1][jc]).sum(0), diag + Cc.sum(0)
        E[l] = _cg(nb[l], torch.where(inner, C, 0.0), diag, rhs, E[l], leaf[l])
        if fld:
            new = T[l] + sigma * (E[l] - T[l] ** 4) / (X[l] * (1 + sigma * mu))
            T[l] = torch.where(leaf[l], new, T[l])

    advance(0, dt0)
    for l in range(n - 2, -1, -1):
        E[l][up[l + 1]] = E[l + 1].reshape(-1, 8).mean(1)
    return E + (T if fld else [])
