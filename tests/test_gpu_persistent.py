"""The persistent Krylov kernel (small sectors: whole steps in one cooperative
launch) against the separate kernels, which a pinned configuration selects,
on the same inputs, and its bounded grid-wide waits.

Tolerances: both sides round a state of unit norm n_steps * m times; for
complex128 300 roundings of 1.1e-16 with a margin of 30 give 1e-12, for
complex64 the roundings are random (no cancellation in a unit-norm state):
sqrt(300) * 6e-8 with a margin of 5 gives 5e-6.  m_eff is the same integer,
except that in complex64 an epsilon within rounding of the adaptive tolerance
(1e-7, two float32 roundings) may take the exit a step earlier or later.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import torch_cuda, to_dev, from_dev, rel_l2, ed_dtype

pytestmark = pytest.mark.gpu

PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0, "dir": (1.0, 1.0, 0.0)}
TOL = {"c128": 1e-12, "c64": 5e-6}
EPS = [0.2, -0.1, 0.0, 0.3, -0.4, 0.1, 0.25, -0.3, 0.15, 0.05, -0.2, 0.35]
PINNED = {"c128": 6, "c64": 3}     # one row per CTA, one kernel per pass


def _eps(lat):
    return dict(lat, eps=np.array(EPS[:lat["Ns"]]))


CASES = [
    (synth.ring(8), 4, 4),               # one row per CTA, fewer rows than SMs
    (_eps(synth.ring(9)), 4, 5),         # 126 rows of 126 columns: two column tiles
    (synth.chain(3), 0, 2),              # one row
    (_eps(synth.chain(3)), 1, 3),        # rows of one column
    (synth.chain(10), 3, 4),             # 120 rows of 210 columns
    (synth.complete_graph(7, seed=3), 3, 4),   # 42 bond groups, odd rows of 35
    (synth.ladder(5), 5, 4),             # 252 rows: two in some CTAs, one in others
    (_eps(synth.torus(4, 3)), 6, 5),     # seven rows in some CTAs, six in others
    (synth.ladder(7), 2, 7),             # 91 rows of 3432 columns
]


def run(ed, torch, h, psi0, dtype, n, m, energy=True):
    x = to_dev(torch, psi0, dtype)
    out = ed.ed_propagate(h.ctx, x, ed_dtype(ed, dtype), PULSE, 0.4, 0.02, n, m, energy=energy)
    torch.cuda.synchronize()
    return from_dev(x), out


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("scheme,tol", [("midpoint", 0.0), ("cfet4", 1e-7)])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_persistent_equals_separate_kernels(ed_lib, case, scheme, tol, dtype):
    torch = torch_cuda()
    ed = ed_lib
    lat, nu, nd = CASES[case]
    h = ed.Hubbard(lat, nu, nd, 6.0)
    ed.ed_set_krylov_tol(h.ctx, tol)
    ed.ed_set_integrator(h.ctx, scheme)
    psi0 = synth.complex_normal(h.D, 5)
    n = 18 if h.D < 100000 else 3        # 18: more than one launch's steps
    m = 14
    try:
        a, oa = run(ed, torch, h, psi0, dtype, n, m)
        b, ob = run(ed, torch, h, psi0, dtype, n, m)
        ed.ed_set_apply_config(PINNED[dtype])
        c, oc = run(ed, torch, h, psi0, dtype, n, m)
    finally:
        ed.ed_set_apply_config(-1)
        h.close()
    assert np.array_equal(a, b)          # sums in a fixed order
    for k in ("docc", "norm2", "energy", "delta"):
        assert np.array_equal(oa[k], ob[k]), k
    assert rel_l2(a, c) <= TOL[dtype]
    if dtype == "c128" or tol == 0.0:
        assert np.array_equal(oa["m_eff"], oc["m_eff"])
    for k in ("docc", "norm2", "energy"):
        assert np.abs(oa[k] - oc[k]).max() <= 10 * TOL[dtype], k
    assert np.abs(oa["delta"] - oc["delta"]).max() <= 10 * TOL[dtype]


def test_persistent_wait_timeout_returns_status_and_context_recovers(ed_lib):
    torch = torch_cuda()
    ed = ed_lib
    lat = synth.ring(8)
    psi0 = synth.complex_normal(4900, 3)
    h = ed.Hubbard(lat, 4, 4, 8.0)
    try:
        ed.ed_set_wait_fault(5, 2000)    # the sixth grid-wide sum of a launch
        x = to_dev(torch, psi0, "c64")
        with pytest.raises(ed.EDError) as e:
            ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, 0.0, 0.02, 2, 6)
        assert e.value.status == 4
        ed.ed_set_wait_fault(-1, 0)
        a, out = run(ed, torch, h, psi0, "c64", 2, 6, energy=False)
        ref = oracle.propagate(lat, 4, 4, 8.0, psi0, PULSE, 0.02, 2, 6, t_start=0.4)
        assert rel_l2(a, ref["psi"]) <= TOL["c64"]
    finally:
        ed.ed_set_wait_fault(-1, 0)
        h.close()
