"""GPU parity of the exact (unprojected) contact Hessian: eipc_contact_hvp and
eipc_eval_contact with EIPC_PARAM_NO_PROJECTION, against the oracle (1e-9 relative), and
the kinematic-position update.

The HVP direction mixes a reduced direction v with a rigid motion of the kinematic
vertices, as the adjoint of a prescribed motion needs.
"""
import dataclasses
import functools

import numpy as np
import pytest

import oracle
from paper_2409_16385_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-9


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@functools.lru_cache(maxsize=None)
def _config1_second_iterate():
    sc = scenes.make_config(1)
    x0 = oracle.embed(sc, sc.iterate(0))
    a = oracle.accd(sc, x0, oracle.embed(sc, sc.dq(0), displacement=True))["alpha"]
    return scenes.with_second_iterate(sc, a)


def _gpu_state(sc, t, lag_t):
    from paper_2409_16385_gb300 import ContactScene
    cs = ContactScene(sc, pair_capacity=1 << 18, bsr_capacity=1 << 19, rec_capacity=1 << 22)
    q, qn = _t(sc.iterate(t)), _t(sc.iterate(lag_t))
    lag = cs.friction_lag(qn, cs.build_candidates(qn, out=cs.new_pairs())) if sc.params["mu"] > 0 else None
    pairs = cs.build_candidates(q)
    return cs, q, pairs, lag


def _oracle_state(sc, t, lag_t, pairs_gpu):
    x = oracle.embed(sc, sc.iterate(t))
    xn = oracle.embed(sc, sc.iterate(lag_t))
    lag = oracle.friction_lag(sc, xn, oracle.pairs(sc, xn)) if sc.params["mu"] > 0 else None
    h = pairs_gpu.host()
    prs = dict(type=h["type"], i=h["i"], j=h["j"])   # same list on both sides (set parity is tested elsewhere)
    return x, prs, lag


def _cases():
    return [("config1", _config1_second_iterate, 1, 0), ("bubble_small", lambda: scenes.make_config(2, small=True), 7, 6)]


@pytest.mark.parametrize("name,make,t,lag_t", _cases())
def test_hvp_matches_oracle(name, make, t, lag_t):
    sc = make()
    cs, q, pairs, lag = _gpu_state(sc, t, lag_t)
    x, prs, lago = _oracle_state(sc, t, lag_t, pairs)
    rng = np.random.default_rng(5)
    kin = sc.kinematic
    for kin_dir in (None, np.array([0.3, -0.2, 1.0])):
        v = rng.normal(size=(sc.Ns, 3))
        out, out_kin = cs.contact_hvp(q, pairs, _t(v), lag=lag, kin_dir=kin_dir)
        torch.cuda.synchronize()
        assert cs.status()["flags"] == 0
        u = oracle.embed(sc, v, displacement=True)
        if kin_dir is not None:
            u[kin] = kin_dir
        ro, rk = oracle.hvp(sc, x, prs, lago, u)
        g = out.cpu().numpy()
        scale = np.abs(ro).max()
        assert scale > 0
        assert np.abs(g - ro).max() <= TOL * scale, (name, np.abs(g - ro).max() / scale)
        gk = out_kin.cpu().numpy()
        if kin.any():
            assert np.abs(gk - rk).max() <= TOL * max(np.abs(rk).max(), 1e-300) + 1e-12 * scale


@pytest.mark.parametrize("name,make,t,lag_t", _cases())
def test_unprojected_hessian_matches_oracle(name, make, t, lag_t):
    sc = make()
    cs, q, pairs, lag = _gpu_state(sc, t, lag_t)
    x, prs, lago = _oracle_state(sc, t, lag_t, pairs)
    E, g, H = cs.eval_contact(q, pairs, lag, project=False)
    torch.cuda.synchronize()
    ro = oracle.eval_contact(sc, x, prs, lago, project=False)
    h = H.host()
    hg = {}
    for r in range(sc.Ns):
        for k in range(h["row_ptr"][r], h["row_ptr"][r + 1]):
            hg[(r, int(h["col"][k]))] = h["val"][k]
    ho = {(int(i), int(j)): vv for i, j, vv in zip(ro["I"], ro["J"], ro["V"])}
    assert set(hg) == set(ho)
    hs = max(np.abs(vv).max() for vv in ho.values())
    assert max(np.abs(hg[k] - ho[k]).max() for k in ho) <= TOL * hs
    # the HVP of the same state equals this matrix times v
    v = np.random.default_rng(9).normal(size=(sc.Ns, 3))
    out, _ = cs.contact_hvp(q, pairs, _t(v), lag=lag)
    ref = np.zeros_like(v)
    for (r, c), B in hg.items():
        ref[r] += B @ v[c]
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    # and the projected Hessian differs (some pair Hessians are indefinite)
    _, _, Hp = cs.eval_contact(q, pairs, lag)
    assert not np.array_equal(Hp.host()["val"], h["val"])


def test_hvp_is_bitwise_repeatable():
    sc = _config1_second_iterate()
    cs, q, pairs, lag = _gpu_state(sc, 1, 0)
    v = _t(np.random.default_rng(2).normal(size=(sc.Ns, 3)))
    outs = [cs.contact_hvp(q, pairs, v, lag=lag, kin_dir=(0.0, 0.0, 1.0)) for _ in range(3)]
    ref = (outs[0][0].cpu().numpy().tobytes(), outs[0][1].cpu().numpy().tobytes())
    for o in outs[1:]:
        assert (o[0].cpu().numpy().tobytes(), o[1].cpu().numpy().tobytes()) == ref


def test_set_kinematic_equals_a_scene_built_with_the_new_positions():
    from paper_2409_16385_gb300 import ContactScene
    sc = scenes.make_config(1)
    shift = np.array([0.0, 0.0, 1e-4])
    kin = sc.kinematic
    moved = dataclasses.replace(sc, x_kin=np.where(kin[:, None], sc.x_kin + shift, sc.x_kin))
    q = _t(sc.iterate(0))
    a = ContactScene(sc, pair_capacity=1 << 18, bsr_capacity=1 << 19, rec_capacity=1 << 22)
    b = ContactScene(moved, pair_capacity=1 << 18, bsr_capacity=1 << 19, rec_capacity=1 << 22)
    a.set_kinematic(_t(moved.x_kin))
    outs = []
    for cs in (a, b):
        pr = cs.build_candidates(q)
        E, g, H = cs.eval_contact(q, pr, None)
        ph = pr.host()
        outs.append((ph["i"].tobytes(), ph["j"].tobytes(), ph["d"].tobytes(), E.cpu().numpy().tobytes(),
                     g.cpu().numpy().tobytes(), H.host()["val"].tobytes()))
        assert cs.status()["flags"] == 0
    assert outs[0] == outs[1]
    assert len(a.build_candidates(q).host()["i"]) > 0


def _point_over_triangle():
    """One contact pair whose Hessian is diagonal in exact arithmetic: a cage node's own vertex over the
    middle of a kinematic triangle, every coordinate a multiple of a power of two."""
    verts = np.array([[0, 0, 0], [2.0**-4, 0, 0], [0, 2.0**-4, 0],
                      [2.0**-6, 2.0**-6, 2.0**-11], [2.0**-6, 2.0**-5, 2.0**-4], [2.0**-5, 2.0**-6, 2.0**-4]])
    idx = np.full((6, 4), -1, np.int32)
    w = np.zeros((6, 4))
    for v in range(3, 6):
        idx[v] = v - 3
        w[v] = 0.25                # no zero weight: its product with an infinity is a NaN
    xk = verts.copy()
    xk[3:] = 0
    tris = np.array([[0, 1, 2], [3, 4, 5]], np.int32)
    return scenes.Scene(name="point_over_triangle", tris=tris, edges=scenes.edges_of(tris), cage_idx=idx, w=w, x_kin=xk, Ns=3,
                        cage_tets=np.zeros((0, 4), np.int32), q_rest=verts[3:].copy(),
                        body=np.array([0, 0, 0, 1, 1, 1], np.int32), params=dict(scenes.DEFAULT_PARAMS))


def test_hvp_components_keep_their_own_precision():
    """A vertex's small components are not held relative to its largest one: with friction along x and
    y and the barrier along z, out's x and y do not change when v's z is raised from 0 to 1, however
    small they are (1e-14: the FP64 operations are the same, the sums lose less)."""
    from paper_2409_16385_gb300 import ContactScene
    sc = _point_over_triangle()
    cs = ContactScene(sc, pair_capacity=64, bsr_capacity=64)
    q = _t(sc.q_rest)
    pairs = cs.build_candidates(q)
    assert pairs.n() == 1
    lag = cs.friction_lag(q, pairs)

    def hvp(x, y, z):
        v = np.zeros((3, 3))
        v[0] = x, y, z
        out, kin = cs.contact_hvp(q, pairs, _t(v), lag=lag)
        return out.cpu().numpy()[0], kin.cpu().numpy()

    one = hvp(0.0, 0.0, 1.0)[0]
    assert one[2] > 0
    for e in (-10, -30, -50, -100, -400):
        a, b = 2.0**e, 3 * 2.0 ** (e - 1)
        alone, beside = hvp(a, b, 0.0)[0], hvp(a, b, 1.0)[0]
        assert alone[0] > 0 and alone[1] > 0 and beside[2] == one[2]
        np.testing.assert_allclose(beside[:2], alone[:2], rtol=1e-14, atol=0)
    # subnormal sums are kept, and a sum beyond FP64's range is infinite
    tiny = hvp(0.0, 0.0, 2.0**-1060)[0]
    np.testing.assert_allclose(tiny[2], one[2] * 2.0**-1060, rtol=2.0**-20, atol=0)
    out, kin = hvp(0.0, 0.0, 4e303)
    assert out[2] == np.inf and kin[2] == -np.inf
    assert cs.status()["flags"] == 0
