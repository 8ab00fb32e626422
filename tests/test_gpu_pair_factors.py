"""The evaluation's pair factors against the oracle on isolated couples of triangles: every
closest-feature class (points, edges, faces), shapes from equilateral to thin, distances from
1e-3 to 0.999 dhat, one to a few hundred pairs (below, at and above a warp's 32), one body
kinematic or both embedded (4 or 8 cage nodes per pair), with and without projection and
friction.  Bars: E to 1e-9 relative, g_r and H_r to 1e-9 of their largest entry, as in the
parity tests; the pattern exactly.
"""
import numpy as np
import pytest

import oracle
from paper_2409_16385_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-9


def couples(n, seed, both):
    """n couples of triangles 2 cm apart, the second a seeded fraction of dhat from the first."""
    rng = np.random.default_rng(seed)
    dhat = scenes.DEFAULT_PARAMS["dhat"]
    b = scenes._Builder()
    side = int(np.ceil(n ** (1.0 / 3.0)))
    for k in range(n):
        o = 0.02 * np.array([k % side, (k // side) % side, k // side ** 2], float)
        A = rng.normal(size=(3, 3)) * dhat * np.array([2.0, 2.0, rng.choice([0.05, 2.0])])
        B = rng.normal(size=(3, 3)) * dhat * 2.0
        gap = dhat * rng.choice([1e-3, rng.uniform(0.05, 0.95), 0.999])
        u = rng.normal(size=3)
        u /= np.linalg.norm(u)
        # slide B along u until the two are `gap` apart (bisection on the oracle's distances)
        def apart(s):
            C = B + s * u
            d2 = [oracle.pair_d2(0, np.array([C[i], *A]))[0] for i in range(3)]
            d2 += [oracle.pair_d2(0, np.array([A[i], *C]))[0] for i in range(3)]
            d2 += [oracle.pair_d2(1, np.array([A[i], A[(i + 1) % 3], C[j], C[(j + 1) % 3]]))[0] for i in range(3) for j in range(3)]
            return np.sqrt(min(d2))
        lo, hi = 0.0, 40.0 * dhat
        B = B + 40.0 * dhat * u
        u = -u
        for s in np.linspace(0.0, 80.0 * dhat, 400):      # the first s at which they come closer than gap
            if apart(s) < gap:
                hi = s
                break
            lo = s
        else:
            hi = lo
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            if apart(mid) > gap:
                lo = mid
            else:
                hi = mid
        B = B + lo * u
        for m, kin in ((A, False), (B, not both)):
            verts = m + o
            tri = np.array([[0, 1, 2]], np.int32)
            if kin:
                b.add_kinematic(verts, tri)
            else:
                nodes, tets, grid = scenes.grid_cage(verts.min(0) - 1e-3, verts.max(0) + 1e-3, (1, 1, 1))
                b.add_embedded(verts, tri, nodes, tets, grid)
    sc = b.scene("couples", dict(scenes.DEFAULT_PARAMS))
    q0 = sc.q_rest + rng.normal(0.0, 1e-7, size=sc.q_rest.shape)
    q1 = q0 + rng.normal(0.0, 2e-7, size=q0.shape)
    return sc, q0, q1


@pytest.mark.parametrize("n,both", [(1, False), (3, True), (31, False), (40, True), (90, False)])
@pytest.mark.parametrize("project", [True, False])
def test_factors_match_the_oracle(n, both, project):
    from paper_2409_16385_gb300 import ContactScene
    sc, q0, q1 = couples(n, 10 * n + both, both)
    cs = ContactScene(sc, pair_capacity=1 << 14, bsr_capacity=1 << 16, rec_capacity=1 << 20)
    t = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    lag = cs.friction_lag(t(q0), cs.build_candidates(t(q0), out=cs.new_pairs()))
    x0, x1 = oracle.embed(sc, q0), oracle.embed(sc, q1)
    po, lo = oracle.pairs(sc, x1), oracle.friction_lag(sc, x0, oracle.pairs(sc, x0))
    for friction in (True, False):
        pairs = cs.build_candidates(t(q1))
        E, g, H = cs.eval_contact(t(q1), pairs, lag if friction else None, project=project)
        torch.cuda.synchronize()
        assert cs.status()["flags"] == 0
        h = pairs.host()
        assert np.array_equal(h["i"], po["i"]) and np.array_equal(h["j"], po["j"]) and len(po["i"]) >= n
        r = oracle.eval_contact(sc, x1, po, lo if friction else None, project=project)
        assert abs(E.item() - r["E"]) <= TOL * abs(r["E"])
        assert np.abs(g.cpu().numpy() - r["g"]).max() <= TOL * np.abs(r["g"]).max()
        hh = H.host()
        rows = np.repeat(np.arange(sc.Ns), np.diff(hh["row_ptr"]))
        o = np.lexsort((r["J"], r["I"]))
        assert np.array_equal(rows, r["I"][o]) and np.array_equal(hh["col"], r["J"][o])
        assert np.abs(hh["val"] - r["V"][o]).max() <= TOL * np.abs(r["V"]).max()
