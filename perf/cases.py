"""The workloads the contact stage is timed on, through its public entry points.

A case is a scene, the state it is in and what is asked of the stage there:
  scene   pad     an icosphere on a rigid pad (a few hundred contacts: latency)
          grasp   a noisy sphere squeezed by two membranes (the bubble gripper)
          rack    a thin plate lowered between rigid tines (near-parallel edges)
          sheets  two nearly parallel sheets (deduplicated set, EE mollifier)
          batch   many independent grasps in one scene, one group each
  op      stage     one Newton iteration: contact set, evaluation, step bound
          step      the first iteration of a time step: the stage and the friction lag
          contacts  the contact set alone (a line search asks for it at every trial)
          eval      the evaluation alone, projected (projected Newton)
          exact     the evaluation alone, unprojected, without friction (full Newton)
          ccd       embedding of the step and its bound
          hvp       the exact Hessian-vector product (adjoints, Krylov solves)
          spmv      the reduced Hessian times a vector (the PCG of a Newton step)
The state is an iterate of the scene's own motion, at a seeded fraction of a step, with a
seeded jitter of the cage nodes, as successive Newton iterates differ.

The buffers are the caller's, sized once with room to spare and zero beyond what a call
writes.  `exact` restates the stage in plain 64-bit torch: contacts by a uniform grid,
derivatives of each pair's energy by automatic differentiation of its closest-feature
distance, 12 x 12 projections by a library eigensolver, index_add for the reduction.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2409_16385_gb300 import ContactScene, binding, scenes

F64 = torch.float64


def listed():
    return [
        # the smallest use: one gripper finger on a pad, a few hundred contacts; a control
        # loop waits for every call
        dict(name="pad_stage", scene="pad", op="stage", level=4, cells=64, pairs=1 << 14, blocks=1 << 14),
        # the adjoint of the same small scene asks for Hessian-vector products
        dict(name="pad_hvp", scene="pad", op="hvp", level=4, cells=64, pairs=1 << 14, blocks=1 << 14),
        # a reduced grasp, as a planner runs many of
        dict(name="small_grasp_stage", scene="grasp", op="stage", body=23, membrane=14, iterate=31, pairs=1 << 16,
             blocks=1 << 16),
        # the headline: one Newton iteration of the full bubble-gripper grasp
        dict(name="grasp_stage", scene="grasp", op="stage", body=71, membrane=45, iterate=31, pairs=1 << 19,
             blocks=1 << 17),
        # its parts, as a line search, a Newton solver and an adjoint call them
        dict(name="grasp_contacts", scene="grasp", op="contacts", body=71, membrane=45, iterate=13, pairs=1 << 19,
             blocks=1 << 17),
        dict(name="grasp_eval", scene="grasp", op="eval", body=71, membrane=45, iterate=46, pairs=1 << 19,
             blocks=1 << 17),
        dict(name="grasp_ccd", scene="grasp", op="ccd", body=71, membrane=45, iterate=22, pairs=1 << 19,
             blocks=1 << 17),
        dict(name="grasp_hvp", scene="grasp", op="hvp", body=71, membrane=45, iterate=22, pairs=1 << 19,
             blocks=1 << 17),
        # the dish rack: the start of a time step, and the unprojected evaluation
        dict(name="rack_step", scene="rack", op="step", nx=150, nz=100, tines=10, around=40, up=50, iterate=40,
             pairs=1 << 17, blocks=1 << 16),
        dict(name="rack_exact", scene="rack", op="exact", nx=149, nz=101, tines=10, around=39, up=51, iterate=61,
             pairs=1 << 17, blocks=1 << 16),
        # the two constraint variants together on the contacts they are for
        dict(name="sheets_mollified", scene="sheets", op="stage", cells=16, pairs=1 << 18, blocks=1 << 14),
        # 256 grasps of uneven size in one scene
        dict(name="batch_stage", scene="batch", op="stage", scenes=256, most=50000, iterate=11, pairs=1 << 18,
             blocks=1 << 19),
    ]


def draw(rng):
    def spread(lo, hi):                       # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["pad", "grasp", "grasp", "grasp", "rack", "rack", "sheets", "batch"])
    ops = ["stage", "step", "contacts", "eval", "exact", "ccd", "hvp"]
    if kind == "pad":
        return dict(scene=kind, op=rng.choice(ops), level=rng.randint(3, 5), cells=spread(17, 131), pairs=1 << 16,
                    blocks=1 << 15)
    if kind == "grasp":
        body = spread(15, 71)
        return dict(scene=kind, op=rng.choice(ops + ["spmv"]), body=body, membrane=max(9, int(body * rng.uniform(0.5, 0.7))),
                    iterate=rng.randint(0, 57), pairs=_pow2(80 * body * body + 4096), blocks=1 << 17)
    if kind == "rack":
        nx = spread(41, 150)
        return dict(scene=kind, op=rng.choice(ops), nx=nx, nz=max(25, int(nx * rng.uniform(0.6, 0.75))),
                    tines=rng.randint(4, 10), around=rng.randint(16, 40), up=rng.randint(20, 50),
                    iterate=rng.randint(0, 79), pairs=1 << 17, blocks=1 << 16)
    if kind == "sheets":
        return dict(scene=kind, op=rng.choice(["stage", "eval", "hvp"]), cells=rng.randint(9, 18), pairs=1 << 18,
                    blocks=1 << 14)
    return dict(scene=kind, op="stage", scenes=spread(3, 24), most=spread(4000, 20000), iterate=rng.randint(0, 50),
                pairs=1 << 17, blocks=1 << 17)


def _pow2(n):
    return 1 << (int(n) - 1).bit_length()


# ------------------------------------------------------------------------------ inputs

def _scene(case):
    return _scene_of(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "op", "iterate", "pairs", "blocks"))))


@functools.lru_cache(maxsize=None)
def _scene_of(key):
    c = dict(key)
    if c["scene"] == "pad":
        return scenes.sphere_on_pad(0, level=c["level"], pad_cells=c["cells"])
    if c["scene"] == "grasp":
        s = c["body"] / 71.0                   # cages keep their nodes per surface vertex
        cage = lambda dims: tuple(max(2, int(round(d * s ** (2.0 / 3.0)))) for d in dims)
        return scenes.bubble_grasp(0, n_body=c["body"], n_mem=c["membrane"], body_cage=cage((10, 11, 11)),
                                   mem_cage=cage((19, 5, 16)))
    if c["scene"] == "rack":
        side = max(6, c["nx"] // 8)
        return scenes.plate_in_rack(0, plate_cells=(c["nx"], c["nz"]), n_tines=c["tines"],
                                    tine_segs=(c["around"], c["up"]), plate_cage=(side, 1, side))
    if c["scene"] == "sheets":
        return scenes.parallel_sheets(0, cells=c["cells"])
    return scenes.batched_grasp(c["scenes"], 0, min_tris=2000, max_tris=c["most"])


def _inputs(case, seed):
    """Iterate, lagged iterate, search direction and Hessian-vector direction (numpy)."""
    sc = _scene(case)
    rng = np.random.default_rng([int(seed), 9])
    t = case.get("iterate", 0)
    u = float(rng.uniform(0.0, 1.0)) if case["scene"] in ("grasp", "rack", "batch") else 0.0
    jitter = rng.normal(0.0, 1e-6, size=(sc.Ns, 3))
    q_n = sc.iterate(sc.lag_of(t)) if t else sc.iterate(0)
    q = sc.iterate(t + u if u else t) + jitter
    if case["scene"] == "sheets":              # the upper sheet slides by a fifth of dhat
        q = q + (sc.iterate(1) - sc.iterate(0)) * rng.uniform(0.2, 1.0)
    dq = sc.dq(t) * (1.0 + rng.normal(0.0, 1e-2, size=(sc.Ns, 1)))
    return dict(q=q, q_n=q_n, dq=dq, v=rng.normal(size=(sc.Ns, 3)))


KIN_DIR = (0.1, -0.3, 1.0)                     # the rigid motion of the kinematic bodies
FACTOR = 1e-3                                  # the EE mollifier's, as in IPC


def prepare(case, seed):
    sc, inp = _scene(case), _inputs(case, seed)
    dev = torch.device("cuda")
    on = lambda a: torch.tensor(a, dtype=F64, device=dev)
    # candidates: the library's default, but what a sizing run asks for in a large batch
    cand = 1 << 25 if case["scene"] == "batch" else 0
    cs = ContactScene(sc, pair_capacity=case["pairs"], bsr_capacity=case["blocks"], cand_capacity=cand)
    if case["scene"] == "batch":
        cs.set_groups(sc.body, sc.n_scenes)
    if case["scene"] == "sheets":
        cs.set_dedup()
        cs.set_mollifier(scenes.embedded_positions(sc, sc.q_rest), FACTOR)
    s = dict(case=case, cs=cs, op=case["op"], q=on(inp["q"]), dq=on(inp["dq"]), v=on(inp["v"]))
    f64 = dict(dtype=F64, device=dev)
    s["pairs"], s["lag"], s["H"] = cs.new_pairs(), cs.new_lag(), cs.new_bsr()
    for b in (s["pairs"], s["lag"], s["H"]):
        for t in vars(b).values():
            t.zero_()
    s["E"], s["g"] = torch.zeros(1, **f64), torch.zeros((sc.Ns, 3), **f64)
    s["x"], s["dx"] = torch.zeros((sc.Nv, 3), **f64), torch.zeros((sc.Nv, 3), **f64)
    s["alpha"], s["n_ccd"] = torch.zeros(1, **f64), torch.zeros(1, dtype=torch.int64, device=dev)
    s["hv"], s["hk"] = torch.zeros((sc.Ns, 3), **f64), torch.zeros(3, **f64)
    if case["scene"] == "batch":
        s["E_groups"], s["alpha_groups"] = torch.zeros(sc.n_scenes, **f64), torch.zeros(sc.n_scenes, **f64)
    op = case["op"]
    if op not in ("step", "exact", "contacts", "ccd"):      # friction lagged earlier in the time step
        q_n = on(inp["q_n"])
        cs.friction_lag(q_n, cs.build_candidates(q_n), out=s["lag"])
    if op != "contacts":                                    # what earlier calls of the iteration left
        cs.build_candidates(s["q"], out=s["pairs"])
    if op == "spmv":
        cs.eval_contact(s["q"], s["pairs"], s["lag"], E=s["E"], g_r=s["g"], H=s["H"])
    flags = cs.status()["flags"]
    if flags & ~64:
        raise RuntimeError("capacity or input: device status %d" % flags)
    return s


def run(s):
    cs, op = s["cs"], s["op"]
    out = {}
    if op in ("stage", "step", "contacts"):
        cs.build_candidates(s["q"], out=s["pairs"])
        out["pairs"] = vars(s["pairs"])
    if op == "step":
        cs.friction_lag(s["q"], s["pairs"], out=s["lag"])
        out["lag"] = vars(s["lag"])
    if op in ("stage", "step", "eval", "exact"):
        cs.eval_contact(s["q"], s["pairs"], None if op == "exact" else s["lag"], E=s["E"], g_r=s["g"], H=s["H"],
                        project=op != "exact")
        out.update(E=s["E"], g=s["g"], H=vars(s["H"]))
        if "E_groups" in s:
            out["E_groups"] = cs.group_energy(out=s["E_groups"])
    if op in ("stage", "step", "ccd"):
        cs.embed(s["q"], out=s["x"])
        cs.embed(s["dq"], out=s["dx"], displacement=True)
        cs.accd_toi(s["x"], s["dx"], alpha=s["alpha"], n_candidates=s["n_ccd"])
        out.update(x=s["x"], dx=s["dx"], alpha=s["alpha"], n_ccd=s["n_ccd"])
        if "alpha_groups" in s:
            out["alpha_groups"] = cs.group_alpha(out=s["alpha_groups"])
    if op == "hvp":
        cs.contact_hvp(s["q"], s["pairs"], s["v"], lag=s["lag"], kin_dir=KIN_DIR, out=s["hv"], out_kin=s["hk"])
        out.update(hv=s["hv"], hk=s["hk"])
    if op == "spmv":
        out["y"] = binding.bsr_spmv(s["H"].row_ptr, s["H"].col, s["H"].val, s["v"], out=s["hv"])
    return out


# contact pairs of a scene, about: per surface vertex (pad: in all; sheets: per cell^4 / dhat^2)
def _contacts_about(case, sc):
    return {"pad": 400, "grasp": 1.7 * sc.Nv * (case.get("body", 71) / 71.0) ** 2, "rack": 0.4 * sc.Nv,
            "sheets": 0.25 * case.get("cells", 0) ** 4, "batch": 94 * case.get("scenes", 0)}[case["scene"]]


def work(case):
    sc = _scene(case)
    n, op = _contacts_about(case, sc), case["op"]
    topology = 12 * sc.F + 8 * sc.E
    embedding = 48 * sc.Nv + 24 * sc.Ns
    hessian = 76 * min(case["blocks"], 20 * sc.Ns)
    lag = 0 if op in ("exact", "contacts", "ccd", "spmv") else 120 * n
    by, fl = 0, 0
    if op in ("stage", "step", "contacts"):    # a distance per contact
        by, fl = by + topology + embedding + 20 * n, fl + 100 * n
    if op in ("stage", "step", "eval", "exact"):    # distance, barrier, eigensolve, blocks
        by, fl = by + embedding + 20 * n + lag + hessian, fl + (2000 if op != "exact" else 1000) * n
    if op in ("stage", "step", "ccd"):
        by, fl = by + topology + 2 * embedding + 96 * sc.Nv, fl + 12 * 7 * sc.Nv
    if op == "hvp":
        by, fl = by + embedding + 20 * n + lag + 48 * sc.Ns, fl + 800 * n
    if op == "spmv":
        by, fl = by + hessian + 48 * sc.Ns, fl + 18 * 20 * sc.Ns
    return dict(bytes=int(by), flops=int(fl))


# ------------------------------------------------------------- the same in plain torch
CHUNK = 1 << 22


def _near(P, Q, h):
    """Index pairs (a, b) with |P_a - Q_b| possibly <= h, by a uniform grid of cell h."""
    lo = torch.minimum(P.min(0).values, Q.min(0).values) - h
    n = ((torch.maximum(P.max(0).values, Q.max(0).values) - lo) / h).floor().long() + 3
    cell = lambda X: ((X - lo) / h).floor().long()
    key = lambda c: (c[:, 0] * n[1] + c[:, 1]) * n[2] + c[:, 2]
    kq, order = torch.sort(key(cell(Q)))
    cp = cell(P)
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            k = key(cp + torch.tensor([dx, dy, 0], device=P.device))
            b, e = torch.searchsorted(kq, k - 1), torch.searchsorted(kq, k + 1, right=True)
            ends = torch.cumsum(e - b, 0)
            a0, done = 0, 0
            while a0 < len(P):
                a1 = max(a0 + 1, int(torch.searchsorted(ends, torch.tensor(done + CHUNK, device=P.device))))
                c = (e - b)[a0:a1]
                ia = torch.repeat_interleave(torch.arange(a0, a1, device=P.device)[:len(c)], c)
                off = torch.arange(len(ia), device=P.device) - torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
                yield ia, order[torch.repeat_interleave(b[a0:a1], c) + off]
                a0, done = min(a1, len(P)), int(ends[min(a1, len(P)) - 1])


def _seg(p, a, b):
    e, w = b - a, p - a
    t = ((w * e).sum(1) / (e * e).sum(1)).clamp(0.0, 1.0)
    r = w - t[:, None] * e
    return (r * r).sum(1), t


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _dot(a, b):
    return (a * b).sum(-1)


def _closest(ty, X):
    """Squared distance, weights c (r = sum c_a x_a) of point-triangle (0) or edge-edge (1)."""
    P = X.shape[0]
    c = torch.zeros((P, 4), dtype=F64, device=X.device)
    rows = torch.arange(P, device=X.device)
    if ty == 0:
        p, a, b, g = X.unbind(1)
        e1, e2, w = b - a, g - a, p - a
        n = _cross(e1, e2)
        nn = _dot(n, n)
        b1, b2 = _dot(_cross(w, e2), n) / nn, _dot(_cross(e1, w), n) / nn
        inside = (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1)
        d_in = _dot(w, n) ** 2 / nn
        c_in = torch.stack([torch.ones_like(b1), -(1 - b1 - b2), -b1, -b2], 1)
        segs = [(0, 1, 2, 1.0), (0, 2, 3, 1.0), (0, 3, 1, 1.0)]
    else:
        a0, a1, g0, g1 = X.unbind(1)
        ea, eb, w = a1 - a0, g1 - g0, a0 - g0
        A, B, C, D, E = _dot(ea, ea), _dot(ea, eb), _dot(eb, eb), _dot(ea, w), _dot(eb, w)
        n = _cross(ea, eb)
        nn = _dot(n, n)
        s, t = (B * E - C * D) / nn, (A * E - B * D) / nn
        inside = (nn > 1e-20 * A * C) & (s >= 0) & (s <= 1) & (t >= 0) & (t <= 1)
        d_in = _dot(w, n) ** 2 / nn
        c_in = torch.stack([1 - s, s, -(1 - t), -t], 1)
        segs = [(0, 2, 3, 1.0), (1, 2, 3, 1.0), (2, 0, 1, -1.0), (3, 0, 1, -1.0)]
    ds, ts = zip(*[_seg(X[:, i], X[:, j], X[:, k]) for i, j, k, _ in segs])
    ds, ts = torch.stack(ds, 1), torch.stack(ts, 1)
    k = ds.argmin(1)
    table = torch.tensor([[i, j, l] for i, j, l, _ in segs], device=X.device)[k]
    sign = torch.tensor([f for *_, f in segs], dtype=F64, device=X.device)[k]
    tk = ts[rows, k]
    c[rows, table[:, 0]] = sign
    c[rows, table[:, 1]] = -sign * (1 - tk)
    c[rows, table[:, 2]] = -sign * tk
    return torch.where(inside, d_in, ds[rows, k]), torch.where(inside[:, None], c_in, c), inside


class _Plain:
    """The scene's arrays on the device, and the stage's quantities at given positions."""

    def __init__(self, case):
        self.case, sc = case, _scene(case)
        self.sc, self.dev = sc, torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda a, d: torch.as_tensor(np.ascontiguousarray(a), dtype=d, device=self.dev)
        self.tris, self.edges, self.idx = t(sc.tris, torch.int64), t(sc.edges, torch.int64), t(sc.cage_idx, torch.int64)
        self.w, self.xk, self.kin = t(sc.w, F64), t(sc.x_kin, F64), t(sc.kinematic, torch.bool)
        self.group = t(sc.body, torch.int64) if case["scene"] == "batch" else None
        self.p = sc.params
        self.moll = None
        if case["scene"] == "sheets":
            xr = t(scenes.embedded_positions(sc, sc.q_rest), F64)
            self.moll = ((xr[self.edges[:, 1]] - xr[self.edges[:, 0]]) ** 2).sum(1)

    def embed(self, q, displacement=False):
        q = torch.as_tensor(q, dtype=F64, device=self.dev)
        x = (self.w[:, :, None] * q[self.idx.clamp_min(0)]).sum(1)
        return torch.where(self.kin[:, None], torch.zeros_like(x) if displacement else self.xk, x)

    def stencil(self, ty, i, j):
        return torch.cat([i[:, None], self.tris[j]], 1) if ty == 0 else torch.cat([self.edges[i], self.edges[j]], 1)

    def _search(self, lo, hi, keep):
        """Over PT and EE pairs, not incident and not all kinematic, with overlapping boxes
        (lo, hi: per vertex): yields (type, i, j, stencil)."""
        parts = [None] if self.group is None else range(self.sc.n_scenes)
        for g in parts:
            inv = lambda prim: torch.arange(len(prim), device=self.dev) if g is None else \
                torch.nonzero(self.group[prim[:, 0]] == g).squeeze(1)
            verts = torch.arange(len(lo), device=self.dev)[:, None]
            sides = {0: (verts, self.tris), 1: (self.edges, self.edges)}
            for ty, (A, B) in sides.items():
                ia, ib = inv(A), inv(B)
                la, ha = lo[A[ia]].amin(1), hi[A[ia]].amax(1)
                lb, hb = lo[B[ib]].amin(1), hi[B[ib]].amax(1)
                h = 0.5 * float((ha - la).max() + (hb - lb).max()) * (1 + 1e-9) + 1e-12
                for a, b in _near(0.5 * (la + ha), 0.5 * (lb + hb), h):
                    ok = ((la[a] <= hb[b]) & (lb[b] <= ha[a])).all(1)
                    a, b = ia[a[ok]], ib[b[ok]]
                    if ty == 1:
                        a, b = a[a < b], b[a < b]
                    v = self.stencil(ty, a, b)
                    na = 1 if ty == 0 else 2
                    ok = (v[:, :na, None] != v[:, None, na:]).all(2).all(1) & ~self.kin[v].all(1)
                    if bool(ok.any()):
                        keep(ty, a[ok], b[ok], v[ok])

    def contacts(self, x, dedup):
        got = {0: [], 1: []}
        dhat = self.p["dhat"]

        def keep(ty, i, j, v):
            d2, c, inside = _closest(ty, x[v] - x[v[:, :1]])
            d = d2.sqrt()
            m = (d < dhat) & (d > 0)
            got[ty].append((i[m], j[m], d[m], c[m], inside[m]))

        self._search(x - 0.5 * dhat * (1 + 1e-9), x + 0.5 * dhat * (1 + 1e-9), keep)
        out = []
        for ty in (0, 1):
            if not got[ty]:
                continue
            i, j, d, c, inside = (torch.cat(z) for z in zip(*got[ty]))
            o = torch.argsort(i * (int(j.max()) + 1 if len(j) else 1) + j)
            out.append((torch.full_like(i, ty)[o], i[o], j[o], d[o], c[o], inside[o]))
        ty, i, j, d, c, inside = (torch.cat(z) for z in zip(*out))
        v = torch.empty((len(i), 4), dtype=torch.int64, device=self.dev)
        for k in (0, 1):
            v[ty == k] = self.stencil(k, i[ty == k], j[ty == k])
        if dedup:                              # the first pair of each realising feature pair
            used = torch.where(c != 0, v, torch.full_like(v, -1))
            na = torch.where(ty == 0, 1, 2)
            left = torch.arange(4, device=self.dev)[None, :] < na[:, None]
            side = lambda m: torch.sort(torch.where(m, used, torch.full_like(v, -1)), 1).values[:, 1:]
            l, r = side(left), side(~left)
            swap = ((l[:, 1] >= 0).long() > (r[:, 1] >= 0).long()) | (((l[:, 1] < 0) & (r[:, 1] < 0)) & (l[:, 2] > r[:, 2]))
            f = torch.cat([torch.where(swap[:, None], r, l), torch.where(swap[:, None], l, r),
                           torch.where(inside, 1 + ty, 0)[:, None]], 1)
            _, inv = torch.unique(f, dim=0, return_inverse=True)
            first = torch.full((int(inv.max()) + 1,), len(i), dtype=torch.int64, device=self.dev)
            first.scatter_reduce_(0, inv, torch.arange(len(i), device=self.dev), "amin")
            k = torch.sort(first).values
            ty, i, j, d, c, inside, v = ty[k], i[k], j[k], d[k], c[k], inside[k], v[k]
        return dict(type=ty, i=i, j=j, d=d, c=c, inside=inside, v=v)

    def mollified(self, P, X):
        """(c, eps) of the mollifier, eps 0 where it does not apply."""
        n = _cross(X[:, 1] - X[:, 0], X[:, 3] - X[:, 2])
        c = _dot(n, n)
        if self.moll is None:
            return c, torch.zeros_like(c)
        ee = P["type"] == 1
        i, j = torch.where(ee, P["i"], 0), torch.where(ee, P["j"], 0)
        eps = FACTOR * self.moll[i] * self.moll[j]
        return c, torch.where(ee & (c < eps), eps, torch.zeros_like(c))

    def lag(self, x, P):
        X = x[P["v"]]
        r = (P["c"][:, :, None] * (X - X[:, :1])).sum(1)
        d, dhat = P["d"], self.p["dhat"]
        b1 = -2 * (d - dhat) * torch.log(d / dhat) - (d - dhat) ** 2 / d
        c, eps = self.mollified(P, X)
        m = torch.where(eps > 0, c * (2 / eps - c / eps ** 2), torch.ones_like(c))
        return dict(v=P["v"], gamma=P["c"], n=r / r.norm(dim=1, keepdim=True), anchor=(P["c"][:, :, None] * X).sum(1),
                    lam=self.p["kappa"] * m * b1.abs())

    def local(self, x, P, project, chunk=16384):
        """Per pair: energy, gradient [12], Hessian [12, 12] of its barrier."""
        dhat, kappa = self.p["dhat"], self.p["kappa"]

        def energy(kind, mollified):
            def f(y, eps):
                a, b, c, d = y[0:3], y[3:6], y[6:9], y[9:12]
                if kind == "face" or kind == "lines":
                    e1, e2, w = (c - b, d - b, a - b) if kind == "face" else (b - a, d - c, a - c)
                    n = _cross(e1, e2)
                    d2 = _dot(w, n) ** 2 / _dot(n, n)
                elif kind == "line":           # the point a against the line b c
                    n = _cross(a - b, c - b)
                    d2 = _dot(n, n) / _dot(c - b, c - b)
                else:
                    d2 = _dot(a - b, a - b)
                dist = torch.sqrt(d2)
                E = -kappa * (dist - dhat) ** 2 * torch.log(dist / dhat)
                if mollified:                  # over the stencil in its own order, carried beside y
                    n = _cross(y[15:18] - y[12:15], y[21:24] - y[18:21])
                    cc = _dot(n, n)
                    E = E * cc * (2 / eps - cc / eps ** 2)
                return E
            return f

        X = x[P["v"]] - x[P["v"][:, :1]]
        n = len(X)
        E = torch.zeros(n, dtype=F64, device=self.dev)
        G, H = torch.zeros((n, 12), dtype=F64, device=self.dev), torch.zeros((n, 12, 12), dtype=F64, device=self.dev)
        nz = (P["c"] != 0).sum(1)
        _, eps = self.mollified(P, X)
        kinds = torch.where(P["inside"], torch.where(P["type"] == 0, 0, 1), torch.where(nz == 3, 2, 3))
        eye = torch.eye(12, dtype=F64, device=self.dev)
        for k, kind in enumerate(("face", "lines", "line", "points")):
            for moll in (False, True):
                sel = torch.nonzero((kinds == k) & ((eps > 0) == moll)).squeeze(1)
                for s in torch.split(sel, chunk) if len(sel) else ():
                    c = P["c"][s]
                    # the stencil's used vertices first; a lone point (weight +-1) before its segment
                    rank = torch.where(c == 0, 3.0, 1.0 - 0.5 * (c.abs() == 1).to(F64)) if k > 1 else torch.zeros_like(c)
                    perm = torch.argsort(rank, dim=1, stable=True)
                    M = eye.reshape(4, 3, 12)[perm].reshape(len(s), 12, 12)      # y = M x
                    if moll:
                        M = torch.cat([M, eye.expand(len(s), 12, 12)], 1)
                    f = energy(kind, moll)
                    g = lambda z, m, e: f(m @ z, e)
                    z = X[s].reshape(-1, 12)
                    E[s] = torch.func.vmap(g)(z, M, eps[s])
                    G[s] = torch.func.vmap(torch.func.grad(g))(z, M, eps[s])
                    h = torch.func.vmap(torch.func.hessian(g))(z, M, eps[s])
                    h = 0.5 * (h + h.transpose(1, 2))
                    if project:
                        lam, V = torch.linalg.eigh(h)
                        h = V @ (lam.clamp_min(0)[:, :, None] * V.transpose(1, 2))
                    H[s] = h
        return E, G, H

    def friction(self, x, L):
        eps, mu = self.p["eps_v"] * self.p["h"], self.p["mu"]
        vs = (L["gamma"][:, :, None] * x[L["v"]]).sum(1) - L["anchor"]
        u = vs - L["n"] * _dot(L["n"], vs)[:, None]
        y2 = _dot(u, u)
        y = y2.sqrt()
        slip = y < eps
        ys = torch.where(y2 > 0, y, torch.ones_like(y))
        f0 = torch.where(slip, -y ** 3 / (3 * eps ** 2) + y2 / eps + eps / 3, y)
        f1 = torch.where(slip, 2 / eps - y / eps ** 2, 1 / ys)
        c2 = torch.where(slip, -y / eps ** 2, -1 / ys) / ys ** 2 * (y2 > 0)
        ml = mu * L["lam"]
        I = torch.eye(3, dtype=F64, device=self.dev)
        F = ml[:, None, None] * (f1[:, None, None] * (I - L["n"][:, :, None] * L["n"][:, None, :])
                                 + c2[:, None, None] * u[:, :, None] * u[:, None, :])
        g = (L["gamma"][:, :, None] * (ml * f1)[:, None, None] * u[:, None, :]).reshape(-1, 12)
        return ml * f0, g, F

    def evaluate(self, x, P, L, project, blocks):
        """E, g_r, the BSR arrays (padded to `blocks` rows) and the per-group energies."""
        ns, dev = self.sc.Ns, self.dev
        E, G, H = self.local(x, P, project)
        v = P["v"]
        if L is not None:
            Ef, Gf, F = self.friction(x, L)
            Hf = torch.einsum("pa,pb,pij->paibj", L["gamma"], L["gamma"], F).reshape(-1, 12, 12)
            E, G, H, v = torch.cat([E, Ef]), torch.cat([G, Gf]), torch.cat([H, Hf]), torch.cat([v, L["v"]])
        node = self.idx[v].reshape(-1, 16)                       # vertex-major
        wt = torch.where(self.kin[v][:, :, None], torch.zeros_like(self.w[v]), self.w[v]).reshape(-1, 16)
        g = torch.zeros((ns + 1, 3), dtype=F64, device=dev)
        g.index_add_(0, node.clamp_min(-1).remainder(ns + 1).reshape(-1),
                     (wt.reshape(-1, 4, 4, 1) * G.reshape(-1, 4, 1, 3)).reshape(-1, 3))
        keys, chunk = [], 16384
        pair_keys = lambda m: torch.where((m[:, :, None] >= 0) & (m[:, None, :] >= 0), m[:, :, None] * ns + m[:, None, :], -1)
        for m in torch.split(node, chunk):
            keys.append(torch.unique(pair_keys(m)))
        keys = torch.unique(torch.cat(keys)) if keys else torch.zeros(0, dtype=torch.int64, device=dev)
        keys = keys[keys >= 0]
        val = torch.zeros((blocks + 1, 9), dtype=F64, device=dev)
        for m, w, h in zip(torch.split(node, chunk), torch.split(wt, chunk), torch.split(H, chunk)):
            k = pair_keys(m)
            at = torch.where(k >= 0, torch.searchsorted(keys, k), blocks)
            hb = h.reshape(-1, 4, 3, 4, 3).permute(0, 1, 3, 2, 4).reshape(-1, 4, 1, 4, 1, 9).expand(-1, 4, 4, 4, 4, 9)
            ww = (w[:, :, None] * w[:, None, :]).reshape(-1, 4, 4, 4, 4, 1)
            val.index_add_(0, at.reshape(-1), (ww * hb).reshape(-1, 9))
        rows = torch.zeros(ns + 1, dtype=torch.int64, device=dev)
        rows[1:] = torch.cumsum(torch.bincount(keys // ns, minlength=ns), 0)
        col = torch.zeros(blocks, dtype=torch.int32, device=dev)
        col[:len(keys)] = (keys % ns).to(torch.int32)
        out = dict(E=E.sum()[None], g=g[:ns], H=dict(row_ptr=rows.to(torch.int32), col=col, val=val[:blocks],
                                                     nnzb=torch.tensor([len(keys)], device=dev)))
        if self.group is not None:
            out["E_groups"] = torch.zeros(self.sc.n_scenes, dtype=F64, device=dev).index_add_(0, self.group[v[:, 0]], E)
        return out

    def hvp(self, x, P, L, v):
        v = torch.as_tensor(v, dtype=F64, device=self.dev)
        u = (self.w[:, :, None] * v[self.idx.clamp_min(0)]).sum(1)
        u = torch.where(self.kin[:, None], torch.tensor(KIN_DIR, dtype=F64, device=self.dev), u)
        _, _, H = self.local(x, P, False)
        y = torch.zeros_like(x)
        y.index_add_(0, P["v"].reshape(-1), torch.einsum("pij,pj->pi", H, u[P["v"]].reshape(-1, 12)).reshape(-1, 3))
        _, _, F = self.friction(x, L)
        Fs = torch.einsum("pij,pj->pi", F, (L["gamma"][:, :, None] * u[L["v"]]).sum(1))
        y.index_add_(0, L["v"].reshape(-1), (L["gamma"][:, :, None] * Fs[:, None, :]).reshape(-1, 3))
        out = torch.zeros((self.sc.Ns, 3), dtype=F64, device=self.dev)
        emb = ~self.kin
        out.index_add_(0, self.idx[emb].reshape(-1), (self.w[emb][:, :, None] * y[emb][:, None, :]).reshape(-1, 3))
        return dict(hv=out, hk=y[self.kin].sum(0))

    def ccd(self, x, dx):
        """Conservative advancement over the pairs whose swept boxes overlap."""
        s, cap, e = self.p["accd_s"], self.p["accd_max_iter"], x + dx
        found = [0, torch.ones((), dtype=F64, device=self.dev)]
        groups = torch.ones(self.sc.n_scenes, dtype=F64, device=self.dev) if self.group is not None else None

        def keep(ty, i, j, v):
            found[0] += len(v)
            X, D = x[v], dx[v]
            R = D - D.mean(1, keepdim=True)
            sp = R.norm(dim=2)
            na = 1 if ty == 0 else 2
            L = sp[:, :na].amax(1) + sp[:, na:].amax(1)
            X = X - X[:, :1]
            d0 = _closest(ty, X)[0].sqrt()
            t = torch.ones_like(L)
            k = torch.nonzero((1 - s) * d0 < L).squeeze(1)       # the others reach t = 1 at once
            d, tk = d0[k], torch.zeros_like(L[k])
            for _ in range(cap):
                if not len(k):
                    break
                tn = tk + (1 - s) * d / L[k]
                t[k] = torch.where(tn >= 1, torch.ones_like(tn), tn)
                go = tn < 1
                k, tk = k[go], tn[go]
                Y = X[k] + R[k] * tk[:, None, None]
                d = _closest(ty, Y - Y[:, :1])[0].sqrt()
                go = d > s * d0[k]
                k, tk, d = k[go], tk[go], d[go]
            # the step bound keeps a margin of 2^-30 below the advancement
            t = torch.where(t < 1, t * (1 - 2.0 ** -30), t)
            found[1] = torch.minimum(found[1], t.min())
            if groups is not None:
                groups.scatter_reduce_(0, self.group[v[:, 0]], t, "amin")

        self._search(torch.minimum(x, e), torch.maximum(x, e), keep)
        out = dict(alpha=found[1][None], n_ccd=torch.tensor([found[0]], device=self.dev))
        if groups is not None:
            out["alpha_groups"] = groups
        return out


def exact(case, seed):
    if case["op"] == "spmv":
        return _exact_spmv(case, seed)
    S, inp, op = _Plain(case), _inputs(case, seed), case["op"]
    dedup = case["scene"] == "sheets"

    def padded(d, names, ints=()):
        out = {}
        for k in names:
            a = d[k]
            z = torch.zeros((case["pairs"],) + tuple(a.shape[1:]), dtype=torch.int32 if k in ints else F64, device=S.dev)
            z[:len(a)] = a.to(z.dtype)
            out[k] = z
        out["count"] = torch.tensor([len(d[names[0]])], device=S.dev)
        return out

    x = S.embed(inp["q"])
    P = S.contacts(x, dedup) if op != "ccd" else None
    L = None
    if op == "step":
        L = S.lag(x, P)
    elif op not in ("exact", "contacts", "ccd"):
        x_n = S.embed(inp["q_n"])
        L = S.lag(x_n, S.contacts(x_n, dedup))
    out = {}
    if op in ("stage", "step", "contacts"):
        out["pairs"] = padded(P, ("type", "i", "j", "d"), ("type", "i", "j"))
    if op == "step":
        out["lag"] = padded(L, ("v", "gamma", "n", "anchor", "lam"), ("v",))
    if op in ("stage", "step", "eval", "exact"):
        out.update(S.evaluate(x, P, L, op != "exact", case["blocks"]))
    if op in ("stage", "step", "ccd"):
        dx = S.embed(inp["dq"], displacement=True)
        out.update(x=x, dx=dx, **S.ccd(x, dx))
    if op == "hvp":
        out.update(S.hvp(x, P, L, inp["v"]))
    return out


def _exact_spmv(case, seed):
    full = exact(dict(case, op="eval"), seed)["H"]
    n, k = len(full["row_ptr"]) - 1, int(full["nnzb"])
    v = torch.as_tensor(_inputs(case, seed)["v"], dtype=F64, device=full["val"].device)
    rows = torch.repeat_interleave(torch.arange(n, device=v.device), full["row_ptr"].long().diff())
    y = torch.zeros((n, 3), dtype=F64, device=v.device)
    return dict(y=y.index_add_(0, rows, torch.einsum("kij,kj->ki", full["val"][:k].reshape(-1, 3, 3), v[full["col"][:k].long()])))
