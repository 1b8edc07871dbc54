"""States of norm zero, alone and in a batch, on device memory that held
not-a-number before: no vector that no pass has written may enter a result.
And the other end: a norm that is not finite."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import torch_cuda, to_dev, from_dev, ed_dtype

pytestmark = pytest.mark.gpu

PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0, "dir": (1.0, 0.0, 0.0)}
PINNED = {"c128": 6, "c64": 3}


class Spoiler:
    """Leaves not-a-number in device memory that the library has freed: a host
    state goes through a device copy of its size."""

    def __init__(self, ed, large):
        self.ed = ed
        self.h = [ed.Hubbard(synth.ring(8), 4, k, 1.0) for k in (1, 2, 3, 4)]
        if large:
            self.h.append(ed.Hubbard(synth.ladder(7), 6, 7, 1.0))

    def run(self):
        for h in self.h:
            x = np.full(h.D, np.nan + 1j * np.nan)
            self.ed.ed_double_occupation(h.ctx, x, self.ed.ED_C128)

    def close(self):
        for h in self.h:
            h.close()


@pytest.mark.parametrize("config", [-1, "pinned"])
@pytest.mark.parametrize("tol", [0.0, 1e-6])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("lat,nu,nd", [(synth.ring(6), 3, 2), (synth.ladder(6), 6, 5)])
def test_zero_state(ed_lib, lat, nu, nd, dtype, tol, config):
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(lat, nu, nd, 4.0)
    ed.ed_set_krylov_tol(h.ctx, tol)
    x = to_dev(torch, np.zeros(h.D, complex), dtype)
    spoil = Spoiler(ed, h.D > 10000)
    try:
        ed.ed_set_apply_config(PINNED[dtype] if config == "pinned" else -1)
        spoil.run()
        o = ed.ed_propagate(h.ctx, x, ed_dtype(ed, dtype), PULSE, 0.0, 0.02, 3, 12, energy=True)
        torch.cuda.synchronize()
    finally:
        ed.ed_set_apply_config(-1)
        spoil.close()
        h.close()
    assert not from_dev(x).any()
    for k in ("docc", "norm2", "energy", "delta"):
        assert not o[k].any(), k


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_batch_with_zero_vectors(ed_lib, dtype):
    """A basis state: c annihilates it on empty sites, c+ on occupied ones."""
    torch = torch_cuda()
    ed = ed_lib
    lat, nu, nd = synth.ring(6), 3, 2
    spoil = Spoiler(ed, False)
    h = ed.Hubbard(lat, nu, nd, 4.0)
    psi = np.zeros(h.D, complex)
    u, d = 7, 4
    psi[u * h.dim_dn + d] = 1.0
    try:
        spoil.run()
        g = ed.ed_spectral_propagate(h.ctx, to_dev(torch, psi, "c128"), ed_dtype(ed, dtype), PULSE,
                                     0.02, 3, 10, 6)
    finally:
        spoil.close()
        h.close()
    words = [oracle.spin_basis(6, nu)[u], oracle.spin_basis(6, nd)[d]]
    tol = 1e-12 if dtype == "c128" else 1e-5
    for create, G in enumerate(g):
        for site in range(6):
            for spin in range(2):
                empty = not (words[spin] >> site) & 1
                lives = empty == bool(create)
                assert abs(abs(G[0, site, spin]) - (1.0 if lives else 0.0)) <= tol
                if not lives:      # c annihilates psi(0), not psi(t): the bra alone is not zero
                    assert np.abs(G[:, site, spin]).max() == 0.0



@pytest.mark.parametrize("config", [-1, "pinned"])
@pytest.mark.parametrize("lat,nu,nd", [(synth.ring(6), 3, 2), (synth.chain(5), 0, 2)])
def test_norm_that_overflows(ed_lib, lat, nu, nd, config):
    """complex64 elements whose squares are infinite: the call fails, and the
    state it leaves shows it."""
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(lat, nu, nd, 4.0)
    x = to_dev(torch, 1e22 * synth.complex_normal(h.D, 3), "c64")
    try:
        ed.ed_set_apply_config(PINNED["c64"] if config == "pinned" else -1)
        with pytest.raises(ed.EDError) as e:
            ed.ed_propagate(h.ctx, x, ed.ED_C64, PULSE, 0.0, 0.02, 3, 12)
        torch.cuda.synchronize()
    finally:
        ed.ed_set_apply_config(-1)
        h.close()
    assert e.value.status == 7
    assert np.isnan(from_dev(x)).all()
