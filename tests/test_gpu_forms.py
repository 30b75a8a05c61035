"""Each form of the FP32 step's passes (direct stores, tensor stores with the
fused column pass, one line per thread) at every line length it has, on
either side of a change of length and with odd and even numbers of columns:
the increments of three steps against the oracle's.  The bars are those of
increments.py."""
import dataclasses

import numpy as np
import pytest
import torch

from increments import INC_MAX_TOL, INC_TOL, dt_for_fraction, increment_errors
from paper_0911_2889_gb300 import inputs

# (N1, N2, K1, K2): columns of 192 .. 1536 points, rows of 2 x 192 .. 2 x 1536
BOXES = [(512, 1024, 63, 127), (512, 1024, 64, 128), (512, 1024, 100, 200), (512, 1024, 127, 255), (1024, 2048, 128, 255),
         (1024, 2048, 255, 256), (2048, 4096, 256, 512), (2048, 4096, 511, 1023)]
_CACHE = {}


def _trajectory(orc, flags, box):
    if box not in _CACHE:
        n1, n2, K1, K2 = box
        p = orc.Params(n1, n2, K1=K1, K2=K2, t0=20.0, flags=flags)
        st = inputs.flat_ic(n1, n2, 31, 1e-4, K1=K1, K2=K2).astype(np.complex64).astype(np.complex128)
        p = dataclasses.replace(p, dt=dt_for_fraction(orc, p, st, 0.0, 0.1))
        traj, s, m, t = [st], st, 0.0, p.t0
        for _ in range(3):
            s, m, t = orc.step(p, s, m, t, 1)
            traj.append(s)
        _CACHE.clear()
        _CACHE[box] = (p, traj, m)
    return _CACHE[box]


@pytest.mark.gpu
@pytest.mark.parametrize("variants", ["1,0", "3,2", "4,3"])
@pytest.mark.parametrize("box", BOXES)
def test_increments_of_every_form(fl, orc, monkeypatch, box, variants):
    monkeypatch.setenv("FLAME_FORCE_VARIANTS", variants)
    monkeypatch.delenv("FLAME_FUSE", raising=False)
    p, traj, m3 = _trajectory(orc, fl.FLAME_NONLINEAR_ONLY, box)
    f = fl.Flame(*box[:2], K1=p.K1, K2=p.K2, prec="fp32", gamma=p.gamma, t0=p.t0, dt=p.dt, flags=p.flags)
    assert fl.flame_fused_steps(f.h) == (variants != "4,3")
    prev = traj[0]
    for n in (1, 2, 3):
        state = torch.from_numpy(fl.box_to_abi(traj[0])).cuda().to(f.cdtype)
        mean, t = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.full((1,), p.t0, dtype=torch.float64, device="cuda")
        f.step(state, mean, t, n)
        got = fl.abi_to_box(state.cpu().numpy()).astype(np.complex128)
        rel, mx = increment_errors(got, prev, traj[n], traj[n - 1], p.K1)
        assert rel < INC_TOL["fp32"] and mx < INC_MAX_TOL["fp32"], (n, rel, mx)
        prev = got
    assert abs(mean.item() - m3) < 2e-5 * abs(m3)
    f.close()
