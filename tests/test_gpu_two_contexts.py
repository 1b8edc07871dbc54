"""Contexts in turn and side by side: a kernel's shared-memory limit is a
property of the process, so a second, smaller sector that uses the same kernel
must leave the first one's launches possible.  The same call on the same
inputs gives the same bits whatever other contexts did in between."""
import threading

import numpy as np
import pytest

import synth
from gpu_util import torch_cuda, to_dev, from_dev, ed_dtype

pytestmark = pytest.mark.gpu

PULSE = {"A0": 0.5, "omega": 8.0, "sigma": 2.0, "t0": 1.0, "dir": (1.0, 1.0, 0.0)}
LARGE = (synth.torus(4, 3), 6, 6)     # rows of 924
SMALL = (synth.ring(8), 4, 4)         # rows of 70


def _step(ed, torch, h, x, dtype, energy):
    o = ed.ed_propagate(h.ctx, x, ed_dtype(ed, dtype), PULSE, 0.4, 0.02, 2, 8, energy=energy)
    torch.cuda.synchronize()
    return o


@pytest.mark.parametrize("dtype,config", [("c64", -1), ("c128", -1), ("c64", 0), ("c64", 2),
                                          ("c128", 6), ("c128", 24)])
def test_propagations_of_two_contexts_in_turn(ed_lib, dtype, config):
    torch = torch_cuda()
    ed = ed_lib
    a, b = ed.Hubbard(*LARGE, 6.0), ed.Hubbard(*SMALL, 6.0)
    va = synth.complex_normal(a.D, 1)
    x, y = to_dev(torch, va, dtype), to_dev(torch, synth.complex_normal(b.D, 2), dtype)
    out = []
    try:
        ed.ed_set_apply_config(config)
        for _ in range(2):
            x.copy_(to_dev(torch, va, dtype))
            o = _step(ed, torch, a, x, dtype, True)
            out.append((from_dev(x), o["energy"]))
            _step(ed, torch, b, y, dtype, True)
    finally:
        ed.ed_set_apply_config(-1)
        a.close()
        b.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("dtype,config", [("c64", 0), ("c64", 1), ("c64", 2), ("c64", 21),
                                          ("c128", 5), ("c128", 17), ("c128", 24)])
def test_products_of_two_contexts_in_turn(ed_lib, dtype, config):
    torch = torch_cuda()
    ed = ed_lib
    a, b = ed.Hubbard(*LARGE, 6.0), ed.Hubbard(*SMALL, 6.0)
    x, y = (to_dev(torch, synth.complex_normal(h.D, 3), dtype) for h in (a, b))
    u, w = torch.zeros_like(x), torch.zeros_like(y)
    code = ed_dtype(ed, dtype)
    out = []
    try:
        ed.ed_set_apply_config(config)
        for _ in range(2):
            u.zero_()
            ed.ed_apply_H(a.ctx, x, u, code)
            torch.cuda.synchronize()
            out.append(from_dev(u))
            ed.ed_apply_H(b.ctx, y, w, code)
            torch.cuda.synchronize()
    finally:
        ed.ed_set_apply_config(-1)
        a.close()
        b.close()
    assert np.array_equal(out[0], out[1])
    assert np.abs(out[0]).max() > 0.0


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_contexts_in_threads(ed_lib, dtype):
    """Each thread its own context, sector and stream; every result as alone."""
    torch = torch_cuda()
    ed = ed_lib
    sectors = [LARGE, SMALL, (synth.ladder(5), 5, 4)]
    alone, got = [None] * 3, [None] * 3

    def work(i, res, repeat):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            h = ed.Hubbard(*sectors[i], 6.0)
            psi = synth.complex_normal(h.D, i)
            for _ in range(repeat):
                x = to_dev(torch, psi, dtype)
                s.synchronize()
                o = ed.ed_propagate(h.ctx, x, ed_dtype(ed, dtype), PULSE, 0.4, 0.02, 4, 8,
                                    energy=True, stream=s)
                s.synchronize()
                r = (from_dev(x), o["energy"])
                res[i] = r if res[i] is None or all(map(np.array_equal, res[i], r)) else "differs"
            h.close()

    for i in range(3):
        work(i, alone, 1)
    threads = [threading.Thread(target=work, args=(i, got, 6)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, g in zip(alone, got):
        assert g is not None and g != "differs"
        assert all(map(np.array_equal, a, g))
