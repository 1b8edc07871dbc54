"""The complex64 kernel configuration of small products on both sides of each
line of its rule, and the product against the one-row configuration.  Both
round each of at most 24 terms of an element a few times: the per-element
bound of the other products."""
import pytest

import synth
from gpu_util import torch_cuda, to_dev, from_dev, max_el, TOL_EL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,nu,nd,nvec,entry", [
    (synth.chain(10), 4, 3, 1, 3),        # 210 rows
    (synth.chain(10), 4, 3, 2, 1),        # 420
    (synth.chain(12), 5, 6, 1, 1),        # 792 rows of 924
    (synth.chain(12), 6, 2, 1, 2),        # 924 rows of 66
    (synth.chain(12), 6, 4, 1, 2),        # 924 rows of 495
    (synth.chain(12), 6, 6, 1, 0),        # 924 rows of 924
    (synth.ladder(7), 4, 4, 1, 0),        # 1001 rows of 1001
    (synth.chain(13), 5, 4, 1, 1),        # 1287 rows of 715
    (synth.ladder(7), 7, 2, 1, 2),        # 3432 rows of 91
])
def test_entry_by_rows_and_columns(ed_lib, lat, nu, nd, nvec, entry):
    torch = torch_cuda()
    ed = ed_lib
    h = ed.Hubbard(lat, nu, nd, 4.0)
    ed.ed_set_field(h.ctx, (0.3, 0.15, 0.0))
    x = to_dev(torch, synth.complex_normal(nvec * h.D, 3), "c64")
    out = []
    try:
        for config in (-1, 3):
            ed.ed_set_apply_config(config)
            w = torch.zeros_like(x)
            ed.ed_apply_H(h.ctx, x, w, ed.ED_C64, nvec=nvec)
            torch.cuda.synchronize()
            if config < 0:
                assert ed.ed_get_apply_config(h.ctx)[1] == entry
            out.append(from_dev(w))
    finally:
        ed.ed_set_apply_config(-1)
        h.close()
    assert max_el(out[0], out[1]) <= 2 * TOL_EL["c64"]
