"""Propagations that run whole steps in one kernel (complex64, sectors that fit
the chip's shared memory).

A call of n steps against n calls of one step, bit by bit: with times that
are exact in binary both run the same sub-steps on the same inputs with the
same coefficients, and a launch of one step has no earlier step whose data a
pass could read.  Then the forms of the kernel that need a tolerance, against
the separate kernels that a pinned configuration selects (tolerances as in
test_gpu_persistent).  Every case first shows that its sector takes this
kernel: with a contribution to the kernel's first grid-wide sum withheld, only
there does a wait run out."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import torch_cuda, to_dev, from_dev, rel_l2

pytestmark = pytest.mark.gpu

PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0, "dir": (1.0, 1.0, 0.0)}
DT = 1.0 / 64.0
T0 = 0.375
TOL = 5e-6
PINNED = 3      # one row per CTA, one kernel per pass


def takes_persistent(ed, torch, h):
    assert h.D < 1 << 20      # no other kernel here has waits to run out
    ed.ed_set_wait_fault(0, 2000)
    try:
        x = to_dev(torch, synth.complex_normal(h.D, 1), "c64")
        ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, T0, DT, 1, 2)
    except ed.EDError as e:
        assert e.status == 4
        return True
    finally:
        ed.ed_set_wait_fault(-1, 0)
    return False


def _eps(lat):
    return dict(lat, eps=np.random.default_rng(0).uniform(-0.4, 0.4, lat["Ns"]))


def _repeated(lat, k):
    """Every bond k times at a k-th of its hopping: the same Hamiltonian."""
    return dict(lat, p=np.repeat(lat["p"], k), q=np.repeat(lat["q"], k),
                t=np.repeat(lat["t"] / k, k), d=np.repeat(lat["d"], k, axis=0))


SECTORS = [
    (synth.ring(8), 4, 4),                # a row in some CTAs, none in others
    (_eps(synth.torus(3, 3)), 4, 5),      # two column tiles
    (synth.chain(7), 3, 3),               # odd rows (35)
    (synth.complete_graph(7, seed=3), 4, 3),   # 42 bond groups
    (synth.ladder(5), 5, 4),              # two rows in some CTAs, one in others
    (synth.chain(12), 4, 4),              # odd rows (495), four in some CTAs
    (synth.torus(4, 3), 6, 5),            # seven rows in some CTAs
    (synth.chain(11), 11, 5),             # one row, one CTA
    (synth.chain(6), 2, 0),               # rows of one column
]


@pytest.mark.parametrize("energy", [False, True])
@pytest.mark.parametrize("m", [2, 9])
@pytest.mark.parametrize("k", range(len(SECTORS)))
def test_steps_equal_calls_of_one_step(ed_lib, k, m, energy):
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(*SECTORS[k], 6.0)
    psi0 = to_dev(torch, synth.complex_normal(h.D, 5), "c64")
    n = 20                                # more than one launch holds
    keys = ("docc", "norm2") + (("energy",) if energy else ())
    try:
        assert takes_persistent(ed, torch, h)
        x = psi0.clone()
        one = {q: [] for q in keys + ("delta", "m_eff")}
        for s in range(n):
            o = ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, T0 + s * DT, DT, 1, m, energy=energy)
            for q in keys:
                one[q] += list(o[q][0 if s == 0 else 1:])
            one["delta"] += list(o["delta"])
            one["m_eff"] += list(o["m_eff"])
        ref = from_dev(x)
        for _ in range(4):
            x.copy_(psi0)
            o = ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, T0, DT, n, m, energy=energy)
            assert np.array_equal(from_dev(x), ref)
            for q in one:
                assert np.array_equal(o[q], np.array(one[q])), q
    finally:
        h.close()


@pytest.mark.parametrize("scheme,n", [("midpoint", 20), ("cfet4", 9)])
@pytest.mark.parametrize("lat,nu,nd", [(synth.torus(4, 3), 6, 5), (_eps(synth.chain(13)), 4, 4),
                                       (synth.chain(12), 6, 4)])
def test_adaptive_exit(ed_lib, lat, nu, nd, scheme, n):
    """Sectors above 2^18 elements, of even and odd row length, over more than
    one launch: the warp that checks beside the passes."""
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(lat, nu, nd, 6.0)
    assert h.D > 1 << 18
    ed.ed_set_integrator(h.ctx, scheme)
    psi0 = synth.complex_normal(h.D, 5)
    m, out = 14, []
    try:
        assert takes_persistent(ed, torch, h)
        ed.ed_set_krylov_tol(h.ctx, 1e-6)
        for config in (-1, -1, PINNED):
            ed.ed_set_apply_config(config)
            x = to_dev(torch, psi0, "c64")
            o = ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, T0, 0.02, n, m, energy=True)
            torch.cuda.synchronize()
            out.append((from_dev(x), o))
    finally:
        ed.ed_set_apply_config(-1)
        h.close()
    (a, oa), (b, ob), (c, oc) = out
    assert np.array_equal(a, b) and np.array_equal(oa["m_eff"], ob["m_eff"])
    assert 2 < oa["m_eff"].min() and oa["m_eff"].max() < m
    assert np.abs(oa["m_eff"] - oc["m_eff"]).max() <= 1
    assert rel_l2(a, c) <= TOL
    for q in ("docc", "norm2", "energy"):
        assert np.abs(oa[q] - oc[q]).max() <= 10 * TOL, q


@pytest.mark.parametrize("rep", [1, 7, 40, 41])
def test_rows_with_many_entries(ed_lib, rep):
    """Up to 8 x 41 entries in a row's list, in numbers that leave every
    remainder of a batch of entries."""
    torch = torch_cuda()
    ed = ed_lib
    lat, nu, nd = synth.chain(6), 3, 2
    pulse = dict(PULSE, dir=(1.0, 0.0, 0.0))
    v = synth.complex_normal(300, 2)
    ref = oracle.propagate(lat, nu, nd, 8.0, v, pulse, 0.02, 3, 10)
    h = ed.Hubbard(_repeated(lat, rep), nu, nd, 8.0)
    try:
        assert takes_persistent(ed, torch, h)
        x = to_dev(torch, v, "c64")
        ed.ed_propagate(h.ctx, x, ed.ED_C64, pulse, 0.0, 0.02, 3, 10)
        torch.cuda.synchronize()
        assert rel_l2(from_dev(x), ref["psi"]) <= TOL
    finally:
        h.close()


def test_room_for_few_steps(ed_lib):
    """182 bond groups and seven rows of 1001 columns in a CTA: with energies
    the shared memory does not hold the coefficients of 16 steps, and a launch
    is given fewer."""
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(synth.complete_graph(14, seed=1), 4, 4, 6.0)
    psi0 = to_dev(torch, synth.complex_normal(h.D, 5), "c64")
    n = 15
    try:
        assert takes_persistent(ed, torch, h)
        x, y = psi0.clone(), psi0.clone()
        o = ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, T0, DT, n, 4, energy=True)
        e = [ed.ed_propagate(h.ctx, y, ed.ED_C64, PULSE, T0 + s * DT, DT, 1, 4, energy=True)
             for s in range(n)]
        assert np.array_equal(from_dev(x), from_dev(y))
        assert np.array_equal(o["energy"][1:], [q["energy"][1] for q in e])
    finally:
        h.close()
