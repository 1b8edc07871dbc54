"""Double occupancies at the sizes where the reduction changes its shape: one
column, one row, rows shorter and longer than a thread block, more rows than a
block's share, all four groups of site bits, and a non-finite element.

Every value is a sum of D products of nonnegative numbers in float64 (the
squares of complex64 elements are exact there), so its rounding is at most
D eps relative to |psi|^2 = 1 in the worst case and about sqrt(D) eps; with a
margin that is 1e-14 for D <= 12870.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import torch_cuda, to_dev, ed_dtype

pytestmark = pytest.mark.gpu

CASES = [(3, 0, 2), (3, 3, 1), (5, 2, 5), (9, 4, 2), (12, 1, 5), (12, 5, 1), (16, 1, 2), (16, 4, 0),
         (16, 8, 0), (16, 0, 8), (16, 15, 14)]


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("Ns,nu,nd", CASES)
def test_double_occupations(ed_lib, Ns, nu, nd, dtype):
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(synth.chain(Ns), nu, nd, 2.0)
    x = to_dev(torch, synth.complex_normal(h.D, 4), dtype)
    code = ed_dtype(ed, dtype)
    d, site = ed.ed_double_occupation(h.ctx, x, code)
    ds, sites = ed.ed_double_occupation_static(h.ctx, x, code)
    q = np.abs(x.cpu().numpy().astype(np.complex128).reshape(h.dim_up, h.dim_dn)) ** 2
    up, dn = ed.ed_get_basis(h.ctx, 0), ed.ed_get_basis(h.ctx, 1)
    for i in range(Ns):
        ref = ((up >> i) & 1).astype(float) @ q @ ((dn >> i) & 1).astype(float)
        assert abs(site[i] - ref) <= 1e-14
    assert abs(d - sum(site[:Ns]) / Ns) <= 1e-14
    assert ds == d and np.array_equal(site, sites)
    # a non-finite element shows in the average wherever it stands
    x[h.D // 2] = float("nan")
    assert np.isnan(ed.ed_double_occupation(h.ctx, x, code)[0])
    h.close()
