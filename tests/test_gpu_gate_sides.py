"""The adaptive exit's step graph, whose passes after the tenth are a conditional
node (from 13 vectors on, 15 in small sectors): exits on each side of the tenth
pass, shown to lie there, the numbers of vectors on each side of those lines,
and a batch whose vectors exit on both sides.  The same passes run on the same
inputs however they are launched, so all results are equal bit by bit."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda, to_dev, from_dev, ed_dtype

pytestmark = pytest.mark.gpu

PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0, "dir": (1.0, 1.0, 0.0)}
PINNED = {"c128": 6, "c64": 3}
TOL = {"c128": 1e-9, "c64": 1e-6}


def _run(ed, torch, dtype, dt, m, profile, sector=(synth.ring(8), 4, 4)):
    h = ed.Hubbard(*sector, 6.0)
    ed.ed_set_krylov_tol(h.ctx, TOL[dtype])
    x = to_dev(torch, synth.complex_normal(h.D, 5), dtype)
    try:
        ed.ed_set_apply_config(PINNED[dtype])
        o = ed.ed_propagate(h.ctx, x, ed_dtype(ed, dtype), PULSE, 0.3, dt, 4, m, energy=True,
                            profile=profile)
        torch.cuda.synchronize()
        return from_dev(x), o
    finally:
        ed.ed_set_apply_config(-1)
        h.close()


@pytest.mark.parametrize("m", [19, 30])
@pytest.mark.parametrize("dtype,dt,least,most", [
    ("c128", 0.01, 3, 9), ("c128", 0.04, 10, 11), ("c128", 0.06, 10, 11), ("c128", 0.14, 13, 18),
    ("c64", 0.02, 3, 9), ("c64", 0.1, 10, 11), ("c64", 0.14, 10, 12), ("c64", 0.2, 12, 18)])
def test_exits_on_each_side(ed_lib, dtype, dt, least, most, m):
    torch = torch_cuda()
    (a, oa), (b, ob) = (_run(ed_lib, torch, dtype, dt, m, p) for p in (True, False))
    assert least <= oa["m_eff"].min() and oa["m_eff"].max() <= most
    assert np.array_equal(a, b)
    for k in ("m_eff", "delta", "docc", "norm2", "energy"):
        assert np.array_equal(oa[k], ob[k]), k


@pytest.mark.parametrize("sector,ms", [((synth.ring(8), 4, 4), (11, 12, 13, 14, 15, 16)),
                                       ((synth.torus(4, 3), 6, 5), (12, 13, 14))])
@pytest.mark.parametrize("dt", [0.02, 0.2])      # an early exit, and none at all
def test_numbers_of_vectors_around_the_lines(ed_lib, dt, sector, ms):
    torch = torch_cuda()
    for m in ms:
        (a, oa), (b, ob) = (_run(ed_lib, torch, "c128", dt, m, p, sector) for p in (True, False))
        assert (oa["m_eff"].max() < 10) if dt < 0.1 else (oa["m_eff"] == m).all()
        assert np.array_equal(a, b)
        for k in ("m_eff", "delta", "docc", "norm2", "energy"):
            assert np.array_equal(oa[k], ob[k]), k


def test_batch_with_exits_on_both_sides(ed_lib):
    """The batch with the conditional node (m = 30) and without (m = 12), for the
    steps whose exits are below 12."""
    torch = torch_cuda()
    ed = ed_lib
    lat = synth.ladder(3)
    psi = synth.complex_normal(225, 5)
    h = ed.Hubbard(lat, 2, 4, 6.0)
    dst = [ed.Hubbard(lat, 2 + c, 4, 6.0) for c in (-1, 1)]
    x = to_dev(torch, psi, "c128")
    phis = [x]
    for q, d in enumerate(dst):
        y = torch.zeros(d.D, dtype=torch.complex128, device="cuda")
        ed.ed_apply_fermion_op(h.ctx, d.ctx, 0, 0, q, x, y, ed.ED_C128)
        phis.append(y)
    ed.ed_set_krylov_tol(h.ctx, TOL["c128"])
    both = 0
    try:
        ed.ed_set_apply_config(PINNED["c128"])
        for dt in (0.08, 0.084, 0.092, 0.1):
            exits = []
            for c, v in zip([h] + dst, phis):
                ed.ed_set_krylov_tol(c.ctx, TOL["c128"])
                o = ed.ed_propagate(c.ctx, v.clone(), ed.ED_C128, PULSE, 0.0, dt, 1, 30)
                exits.append(int(o["m_eff"][0]))
            if max(exits) >= 12:
                continue
            both += min(exits) <= 10 < max(exits)
            g = [ed.ed_spectral_propagate(h.ctx, x, ed.ED_C128, PULSE, dt, 1, m, 6)
                 for m in (30, 12)]
            for u, v in zip(*g):
                assert np.array_equal(u, v)
    finally:
        ed.ed_set_apply_config(-1)
        for c in [h] + dst:
            c.close()
    assert both > 0
