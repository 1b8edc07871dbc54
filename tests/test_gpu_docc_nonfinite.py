"""Double occupancies of states with elements that are not finite, or whose
square is not: the sites that weigh such an element show it, the others keep
their values, and the average is the sum over all elements of (doubly occupied
sites) |psi|^2, in which 0 times infinity is not a number."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda, to_dev, ed_dtype

pytestmark = pytest.mark.gpu

LAT, NU, ND = synth.chain(7), 3, 2


def _words(n, k):
    return np.array([w for w in range(1 << n) if bin(w).count("1") == k])


def _expected(psi):
    both = _words(7, NU)[:, None] & _words(7, ND)[None, :]
    q = (psi.real ** 2 + psi.imag ** 2).reshape(both.shape)
    n = np.zeros(both.shape)
    site = np.zeros(7)
    for i in range(7):
        m = (both >> i) & 1 == 1
        site[i] = q[m].sum()
        n += m
    return (n * q).sum() / 7, site


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e200])
@pytest.mark.parametrize("sites", [0, 1, 2])
def test_elements_that_are_not_finite(ed_lib, sites, value, dtype):
    torch = torch_cuda()
    ed = ed_lib
    if value == 1e200 and dtype == "c64":
        pytest.skip("an infinity in complex64")
    h = ed.Hubbard(LAT, NU, ND, 4.0)
    psi = synth.complex_normal(h.D, 4)
    both = (_words(7, NU)[:, None] & _words(7, ND)[None, :]).reshape(-1)
    at = [t for t in range(h.D) if bin(both[t]).count("1") == sites][5]
    psi[at] = complex(value, 0.25)
    x = to_dev(torch, psi, dtype)
    with np.errstate(all="ignore"):
        avg, site = _expected(x.cpu().numpy().astype(np.complex128))
    try:
        ref = ed.ed_double_occupation(h.ctx, x, ed_dtype(ed, dtype))
        stat = ed.ed_double_occupation_static(h.ctx, x, ed_dtype(ed, dtype))
    finally:
        h.close()
    for d, s in (ref, stat):
        np.testing.assert_allclose(s[:7], site, rtol=1e-13)
        np.testing.assert_allclose(d, avg, rtol=1e-13)
    assert not np.isfinite(avg)
