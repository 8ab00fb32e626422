"""Record workspace too small for an evaluation: factor rows (one per item and cage node) past the row
workspace, explicit records of mollified pairs past the record workspace, and both.  The call raises
REC_OVERFLOW with the size needed and leaves the energy whole; a scene of that size gives the bits
of one with room to spare.  Two sheets: 6,628 pairs, 34,962 rows, 112,770 records without friction.
"""
import numpy as np
import pytest

import oracle
from paper_2409_16385_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CAND = 1 << 14          # room for the 12,324 candidates and 13,256 items, but for fewer rows than any case has


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _evaluate(sc, xr, moll, lagged, rec):
    from paper_2409_16385_gb300 import ContactScene
    cs = ContactScene(sc, pair_capacity=1 << 13, bsr_capacity=1 << 16, cand_capacity=CAND, rec_capacity=rec)
    if moll:
        cs.set_mollifier(xr)
    q0, q1 = _t(sc.iterate(0)), _t(sc.iterate(1))
    lag = cs.friction_lag(q0, cs.build_candidates(q0, out=cs.new_pairs())) if lagged else None
    pairs = cs.build_candidates(q1)
    assert cs.status()["flags"] == 0
    E, g, H = cs.eval_contact(q1, pairs, lag)
    return cs, E.item(), g.cpu().numpy(), H.host(), cs.status()


@pytest.mark.parametrize("moll,lagged,rec", [(False, False, 1000), (False, True, 1000), (True, False, 1000),
                                             (True, True, 1000), (True, False, 60000), (True, False, 112769)])
def test_overflow_is_reported_and_a_scene_of_the_size_needed_is_whole(moll, lagged, rec):
    sc = scenes.parallel_sheets()
    xr = oracle.embed(sc, sc.q_rest)
    _, E0, g0, H0, st = _evaluate(sc, xr, moll, lagged, 1 << 22)
    assert st["flags"] == 0
    cs, E1, _, _, st = _evaluate(sc, xr, moll, lagged, rec)
    assert "REC_OVERFLOW" in st["names"] and st["needed"][2] > rec
    assert E1 == E0
    assert cs.build_candidates(_t(sc.iterate(0))).n() > 0 and cs.status()["flags"] == 0      # the scene goes on
    _, E2, g2, H2, st2 = _evaluate(sc, xr, moll, lagged, st["needed"][2])
    assert st2["flags"] == 0 and E2 == E0
    np.testing.assert_array_equal(g2, g0)
    for k in ("row_ptr", "col", "val"):
        np.testing.assert_array_equal(H2[k], H0[k])


def test_deduplication_reports_the_pairs_it_has_no_room_for():
    from paper_2409_16385_gb300 import ContactScene
    sc = scenes.parallel_sheets()
    q, got = _t(sc.iterate(1)), {}
    for rec in (1 << 22, 1000, 6628):
        cs = ContactScene(sc, pair_capacity=1 << 13, bsr_capacity=1 << 16, cand_capacity=CAND, rec_capacity=rec)
        cs.set_dedup()
        h = cs.build_candidates(q).host()
        st = cs.status()
        if rec == 1000:
            assert st["names"] == ["REC_OVERFLOW"] and st["needed"][2] == 6628
        else:
            assert st["flags"] == 0
            got[rec] = [h[k].tobytes() for k in ("type", "i", "j", "d")]
    assert got[1 << 22] == got[6628]
