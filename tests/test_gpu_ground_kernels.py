"""Ground-state solve at the sizes where its kernels change their shape:
one element, fewer elements than a thread block, chunks with a remainder, many
restarts with few vectors, and a host result.

H y = E y is checked with ed_apply_H; the energy against the oracle.  The
solve stops at a residual of tol max(1, |E|), so that is the tolerance of the
residual (with a factor of 2 for the product's own rounding) and, by the
Temple bound, more than that of the energy.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

EPS = np.array([0.2, -0.1, 0.0, 0.3, -0.4, 0.1, 0.25, -0.3])

CASES = [
    (synth.chain(2), 0, 2, 0, 0),        # one element
    (synth.chain(3), 0, 2, 0, 0),        # three elements
    (synth.chain(5), 2, 1, 0, 0),        # 50 elements: part of one block
    (synth.ring(8), 4, 3, 0, 0),         # 3920 elements: chunks of 1024 with a remainder
    (synth.ring(8), 4, 3, 0, 23),        # restarts with 20 Lanczos vectors
    (synth.torus(3, 3), 4, 5, 1, 0),     # 15876 elements, result in host memory
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_ground_state_sizes(ed_lib, case):
    torch = torch_cuda()
    ed = ed_lib
    lat, nu, nd, host, limit = CASES[case]
    lat = dict(lat, eps=EPS[:lat["Ns"]] if lat["Ns"] <= 8 else None)
    h = ed.Hubbard(lat, nu, nd, 5.0)
    if limit:
        ed.ed_set_workspace_limit(h.ctx, limit * 16 * h.D)
    psi = np.zeros(h.D, np.complex128) if host else torch.zeros(h.D, dtype=torch.complex128,
                                                                device="cuda")
    tol = 1e-10
    E, res = ed.ed_ground_state(h.ctx, psi, tol=tol, max_iter=6000, seed=3)
    assert res <= tol * max(1.0, abs(E))
    x = torch.from_numpy(psi).cuda() if host else psi
    w = torch.zeros_like(x)
    ed.ed_apply_H(h.ctx, x, w, ed.ED_C128)
    torch.cuda.synchronize()
    v = x.cpu().numpy()
    assert np.linalg.norm(w.cpu().numpy() - E * v) <= 2 * tol * max(1.0, abs(E))
    assert abs(np.linalg.norm(v) - 1.0) <= 1e-13
    k = int(np.argmax(np.abs(v)))
    assert abs(v[k].imag) <= 1e-13 and v[k].real > 0
    H = oracle.build_H(lat, nu, nd, 5.0)
    E0 = np.linalg.eigvalsh(H.toarray())[0] if h.D < 4000 else oracle.ground_state(lat, nu, nd, 5.0)[0]
    assert abs(E - E0) <= tol * max(1.0, abs(E0))
    h.close()
