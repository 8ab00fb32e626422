"""Contact sets over every form of the hierarchies and of their walk, against the oracle: trees of
one leaf, of one treelet (32 leaves) and one more, of one cluster (512) and one more, the largest
scene refitted by clusters (2^20 triangles and edges) and one beyond it; spread evenly, in tight
groups a metre apart (one walk spans several), and with one primitive so far away that the rest
share a Morton cell and a warp's queries lie anywhere (the one-node walk).  The pair lists are
compared exactly, after a build and after a refit.
"""
import numpy as np
import pytest

import oracle
from paper_2409_16385_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SIDE = 4.0e-3          # of a triangle's neighbourhood: a few triangles within dhat = 1e-3


def soup(F, layout, seed):
    """F separate triangles; every other one kinematic, the rest embedded in one tetrahedron."""
    rng = np.random.default_rng(seed)
    L = 100.0
    box = SIDE * F ** (1.0 / 3.0)
    c = rng.uniform(0.0, box, size=(F, 3))
    if layout == "groups":
        c = SIDE * rng.uniform(0.0, max(1.0, (F / 40.0) ** (1.0 / 3.0)), size=(F, 3)) + rng.integers(0, 4, size=(F, 3))
    if layout == "outlier" and F > 1:
        c[-1] = 0.3 * L
    x = (c[:, None, :] + rng.normal(size=(F, 3, 3)) * 1.0e-3 + 0.01).reshape(-1, 3)
    tris = np.arange(3 * F, dtype=np.int32).reshape(F, 3)
    kin = np.repeat(np.arange(F) % 2 == 1, 3)
    idx = np.tile(np.arange(4, dtype=np.int32), (3 * F, 1))
    w = np.concatenate([1.0 - x.sum(1, keepdims=True) / L, x / L], axis=1)
    idx[kin] = -1
    w[kin] = 0.0
    q = np.concatenate([np.zeros((1, 3)), L * np.eye(3)])
    sc = scenes.Scene(name="soup", tris=tris, edges=scenes.edges_of(tris), cage_idx=np.ascontiguousarray(idx),
                      w=np.ascontiguousarray(w), x_kin=np.where(kin[:, None], x, 0.0), Ns=4,
                      cage_tets=np.array([[0, 1, 2, 3]], np.int32), q_rest=q, body=np.zeros(3 * F, np.int32),
                      params=dict(scenes.DEFAULT_PARAMS))
    return sc, q, q + rng.normal(0.0, 3e-4, size=(1, 3))


FORMS = [(1, "even"), (2, "even"), (10, "even"), (11, "groups"), (32, "even"), (33, "outlier"), (170, "groups"),
         (171, "even"), (513, "outlier"), (3000, "groups"), (3000, "outlier"), (20000, "even"), (262100, "even"),
         (262200, "groups")]


@pytest.mark.parametrize("F,layout", FORMS)
def test_contact_set_matches_the_oracle(F, layout):
    from paper_2409_16385_gb300 import ContactScene
    sc, q0, q1 = soup(F, layout, F)
    cs = ContactScene(sc, pair_capacity=1 << 16 if F < 10000 else 1 << 22, cand_capacity=1 << 20 if F < 10000 else 1 << 25)
    rng = np.random.default_rng(F)
    found = 0
    for q in (q0, q1):                       # a build, then a refit
        pr = cs.build_candidates(torch.from_numpy(q).cuda()).host()
        assert cs.status()["flags"] == 0
        x = oracle.embed(sc, q)
        if F < 10000:
            po = oracle.pairs(sc, x)
            for k in ("type", "i", "j"):
                np.testing.assert_array_equal(pr[k], po[k])
            found += len(po["type"])
            continue
        for ptype, n in ((0, sc.Nv), (1, sc.E)):         # the pairs of a sample of vertices and edges
            some = np.sort(rng.choice(n, 500, replace=False)).astype(np.int32)
            po = oracle.pairs_of(sc, x, ptype, some)
            mine = (pr["type"] == ptype) & (np.isin(pr["i"], some) | ((ptype == 1) & np.isin(pr["j"], some)))
            want = {(min(a, b), max(a, b)) if ptype else (a, b) for a, b in zip(po["i"].tolist(), po["j"].tolist())}
            assert set(zip(pr["i"][mine].tolist(), pr["j"][mine].tolist())) == want
            found += len(want)
    assert found > 0 or F < 11
