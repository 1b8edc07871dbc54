"""ed_ground_state into result buffers of every kind: the same bits in a device
buffer at a 16-byte boundary, at an odd multiple of 8 bytes, and on the host
(pageable and pinned)."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,nu,nd", [(synth.ring(6), 3, 3), (synth.chain(3), 0, 2),
                                       (synth.chain(2), 0, 0),
                                       (synth.dimer(), 1, 1), (synth.chain(5), 1, 0)])
def test_result_buffers(ed_lib, lat, nu, nd):
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(lat, nu, nd, 4.0)
    n = 2 * h.D
    try:
        host = np.zeros(h.D, np.complex128)
        E, res = ed.ed_ground_state(h.ctx, host, tol=1e-10, max_iter=500, seed=3)
        ref = host.view(np.float64)
        assert abs(np.linalg.norm(ref) - 1.0) <= 1e-12
        pinned = torch.zeros(n, dtype=torch.float64).pin_memory()
        buf = torch.full((n + 4,), 7.0, dtype=torch.float64, device="cuda")
        assert buf.data_ptr() % 16 == 0
        for p, view in ((pinned.data_ptr(), pinned), (buf.data_ptr(), buf[:n]),
                        (buf.data_ptr() + 8, buf[1:1 + n])):
            buf.fill_(7.0)
            torch.cuda.synchronize()
            E2, res2 = ed.ed_ground_state(h.ctx, p, tol=1e-10, max_iter=500, seed=3)
            assert (E2, res2) == (E, res)
            assert np.array_equal(view.cpu().numpy(), ref)
        b = buf.cpu().numpy()
        assert b[0] == 7.0 and (b[1 + n:] == 7.0).all()
    finally:
        h.close()
