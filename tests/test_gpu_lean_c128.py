"""The complex128 products that walk T_dn and T_up together by bond group
(one row per CTA, one kernel), where the walk changes its course: no field
(all coefficients equal, one sum), a field along one direction (some real),
along both, many classes, and rows with more T_up entries than are kept in
shared memory.  Tolerance as for every other product: 1e-13."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import torch_cuda, to_dev, from_dev, rel_l2, max_el

pytestmark = pytest.mark.gpu


def _repeated(lat, k):
    """Every bond k times at a k-th of its hopping: the same Hamiltonian."""
    return dict(lat, p=np.repeat(lat["p"], k), q=np.repeat(lat["q"], k),
                t=np.repeat(lat["t"] / k, k), d=np.repeat(lat["d"], k, axis=0))


LATS = [(synth.ladder(4), 4, 3, 1), (synth.torus(3, 3), 4, 5, 1),
        (synth.complete_graph(6, seed=2), 3, 2, 1), (synth.ring(8), 4, 4, 40),
        (synth.chain(4), 0, 2, 1), (synth.chain(4), 4, 3, 1)]


def lean_configs(ed):
    out = []
    for i in range(ed.ed_apply_config_count()):
        c = ed.ed_apply_config_info(i)
        if c["fp64"] and c["rows_per_cta"] == 1 and not (c["split"] or c["tma"] or c["mv"]):
            out.append(i)
    assert len(out) == 3
    return out


@pytest.mark.parametrize("A", [(0.0, 0.0, 0.0), (0.4, 0.0, 0.0), (0.4, 0.7, 0.0), (0.3, 0.3, 0.0)])
@pytest.mark.parametrize("k", range(len(LATS)))
def test_products_match_oracle(ed_lib, k, A):
    torch = torch_cuda()
    ed = ed_lib
    lat, nu, nd, rep = LATS[k]
    H = oracle.build_H(lat, nu, nd, 3.0, np.array(A))
    h = ed.Hubbard(_repeated(lat, rep), nu, nd, 3.0)
    v = synth.complex_normal(h.D, 7)
    ref = H @ v
    ed.ed_set_field(h.ctx, A)
    try:
        for cfg in lean_configs(ed) + [-1]:
            ed.ed_set_apply_config(cfg)
            x = to_dev(torch, v, "c128")
            w = torch.zeros_like(x)
            ed.ed_apply_H(h.ctx, x, w, ed.ED_C128)
            torch.cuda.synchronize()
            assert rel_l2(from_dev(w), ref) <= 1e-13
            assert max_el(from_dev(w), ref) <= 1e-13
    finally:
        ed.ed_set_apply_config(-1)
        h.close()


def test_repeated_bonds_in_the_persistent_kernel(ed_lib):
    torch = torch_cuda()
    ed = ed_lib
    lat = synth.ring(8)
    pulse = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 0.2, "dir": (1.0, 0.0, 0.0)}
    v = synth.complex_normal(4900, 2)
    ref = oracle.propagate(lat, 4, 4, 8.0, v, pulse, 0.02, 3, 10)
    h = ed.Hubbard(_repeated(lat, 40), 4, 4, 8.0)
    x = to_dev(torch, v, "c128")
    ed.ed_propagate(h.ctx, x, ed.ED_C128, pulse, 0.0, 0.02, 3, 10)
    torch.cuda.synchronize()
    assert rel_l2(from_dev(x), ref["psi"]) <= 1e-10
    h.close()
