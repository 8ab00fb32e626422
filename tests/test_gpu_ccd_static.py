"""eipc_accd_toi_static gives eipc_accd_toi's bound bit for bit: many scenes and motions, a list longer
than the chunks it is taken in, edges that are not aligned to eight bytes, incident and out-of-range
candidates among them."""
import ctypes

import numpy as np
import pytest

from paper_2409_16385_gb300 import binding, scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CHUNK = 1 << 18
MAKE = {"pad": lambda: scenes.make_config(1), "grasp": lambda: scenes.make_config(2, small=True),
        "rack": lambda: scenes.make_config(3, small=True), "sheets": scenes.parallel_sheets}


def _static(sc, x, dx, cand, edges):
    lib, P = binding.load(), ctypes.c_void_p
    lib.eipc_accd_toi_static.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int64, P, P, P, P, ctypes.c_int64,
                                         P, P, P, ctypes.POINTER(binding.Params), P, P, P, P]
    lib.eipc_accd_toi_static.restype = ctypes.c_int32
    tris = torch.tensor(sc.tris, dtype=torch.int32, device="cuda")
    alpha = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    flags = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    nadv = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    params = binding.make_params(sc.params)
    ct, ci, cj = cand
    rc = lib.eipc_accd_toi_static(sc.Nv, sc.F, sc.E, x.data_ptr(), dx.data_ptr(), tris.data_ptr(), edges.data_ptr(), ct.shape[0],
                                  ct.data_ptr(), ci.data_ptr(), cj.data_ptr(), ctypes.byref(params), alpha.data_ptr(),
                                  flags.data_ptr(), nadv.data_ptr(), P(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    return alpha.item(), int(flags.item()), int(nadv.item())


@pytest.mark.parametrize("name", sorted(MAKE))
def test_static_bound_has_the_bits_of_the_scenes(name):
    from paper_2409_16385_gb300 import ContactScene
    sc = MAKE[name]()
    cs = ContactScene(sc, pair_capacity=1 << 18, bsr_capacity=1 << 18, rec_capacity=1 << 20)
    q = torch.tensor(sc.iterate(0), dtype=torch.float64, device="cuda")
    x = cs.embed(q)
    step = cs.embed(torch.tensor(sc.dq(0), dtype=torch.float64, device="cuda"), displacement=True)
    rng = np.random.default_rng(17)
    words = torch.empty(2 * sc.E + 1, dtype=torch.int32, device="cuda")
    words[1:] = torch.tensor(sc.edges, dtype=torch.int32, device="cuda").reshape(-1)
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    bounds = set()
    for k in range(24):
        dx = float(rng.uniform(0.2, 2.0)) * step + torch.tensor(rng.normal(size=(sc.Nv, 3)) * 1e-4, device="cuda")
        a = cs.accd_toi(x, dx, n_candidates=n).item()
        flags = cs.status()["flags"]
        cand = tuple(c.clone() for c in cs.candidates())
        got = _static(sc, x, dx, cand, words[1:])
        assert got == (a, flags, int(n.item())), k
        bounds.add(a)
    assert len(bounds) > 12
    # the same list over and over, past a chunk's end, with candidates that are skipped
    m = cand[0].shape[0]
    times = CHUNK // m + 2
    ct, ci, cj = (c.repeat(times) for c in cand)
    bad = torch.tensor([[0, 0, sc.F], [1, -1, 0], [2, 0, 0], [1, 0, 0]], dtype=torch.int32, device="cuda").T
    ct, ci, cj = (torch.cat([c, b]).contiguous() for c, b in zip((ct, ci, cj), bad))
    assert ct.shape[0] > CHUNK
    assert _static(sc, x, dx, (ct, ci, cj), words[1:]) == (a, flags | 512, times * int(n.item()))
