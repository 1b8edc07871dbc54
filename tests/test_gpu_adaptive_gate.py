"""The adaptive exit's step graph holds the passes after the tenth in a
conditional node.  Exits before it, around it and far behind it against the
profile mode, which launches every pass and check one by one: the same kernels
in the same order on the same inputs, so the results are equal bit by bit."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda, to_dev, from_dev, ed_dtype

pytestmark = pytest.mark.gpu

PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0, "dir": (1.0, 1.0, 0.0)}
PINNED = {"c128": 6, "c64": 3}


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-9), ("c64", 1e-5)])
@pytest.mark.parametrize("dt", [0.01, 0.02, 0.03, 0.04, 0.05, 0.2])
def test_gated_graph_equals_single_launches(ed_lib, dt, dtype, tol):
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(synth.torus(3, 3), 4, 5, 8.0)
    ed.ed_set_krylov_tol(h.ctx, tol)
    psi0 = synth.complex_normal(h.D, 9)
    out = []
    try:
        ed.ed_set_apply_config(PINNED[dtype])
        for profile in (True, False):
            x = to_dev(torch, psi0, dtype)
            o = ed.ed_propagate(h.ctx, x, ed_dtype(ed, dtype), PULSE, 0.3, dt, 3, 30, energy=True,
                                profile=profile)
            torch.cuda.synchronize()
            out.append((from_dev(x), o))
    finally:
        ed.ed_set_apply_config(-1)
        h.close()
    (a, oa), (b, ob) = out
    assert np.array_equal(a, b)
    for k in ("m_eff", "delta", "docc", "norm2", "energy"):
        assert np.array_equal(oa[k], ob[k]), k


def test_breakdown_before_the_gate(ed_lib):
    """A sector of four states: the Krylov space ends at four vectors."""
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(synth.dimer(), 1, 1, 4.0)
    ed.ed_set_krylov_tol(h.ctx, 1e-14)
    x = to_dev(torch, synth.complex_normal(4, 2), "c128")
    try:
        ed.ed_set_apply_config(PINNED["c128"])
        o = ed.ed_propagate(h.ctx, x, ed.ED_C128, None, 0.0, 0.3, 5, 30)
        torch.cuda.synchronize()
    finally:
        ed.ed_set_apply_config(-1)
        h.close()
    assert o["m_eff"].max() <= 4 and np.abs(o["norm2"] - 1.0).max() <= 1e-13
