"""Pass C on either side of the rule that gives it two or three CTAs per SM
(columns of 3072 points, more than four tiles per SM): grids of one wave, of
less than two and of more, a step's increment against the oracle.  The bars
are those of increments.py.  A step on host buffers launches pass C in eight
parts, which are small enough for two: it gives the same bits."""
import dataclasses

import numpy as np
import pytest
import torch

from increments import INC_MAX_TOL, INC_TOL, dt_for_fraction, increment_errors
from paper_0911_2889_gb300 import inputs


@pytest.mark.gpu
@pytest.mark.parametrize("n2,K2", [(64, 0), (2048, 510), (4096, 0), (8192, 1500)])
def test_pass_c_at_either_occupancy(fl, orc, monkeypatch, n2, K2):
    monkeypatch.setenv("FLAME_FORCE_VARIANTS", "1,0")
    n1, flags = 4096, fl.FLAME_NONLINEAR_ONLY
    p = orc.Params(n1, n2, K2=K2, t0=20.0, flags=flags)
    st = inputs.flat_ic(n1, n2, 29, 1e-4, K1=p.K1, K2=p.K2).astype(np.complex64).astype(np.complex128)
    p = dataclasses.replace(p, dt=dt_for_fraction(orc, p, st, 0.0, 0.5))
    ref, mref, _ = orc.step(p, st, 0.0, p.t0, 1)
    f = fl.Flame(n1, n2, K1=p.K1, K2=p.K2, prec="fp32", gamma=p.gamma, t0=p.t0, dt=p.dt, flags=flags)
    state = torch.from_numpy(fl.box_to_abi(st)).cuda().to(f.cdtype)
    mean, t = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.full((1,), 20.0, dtype=torch.float64, device="cuda")
    host = [x.cpu().pin_memory() for x in (state, mean, t)]
    f.step(state, mean, t, 1)
    f.step_host(*host, 1)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b.cpu()) for a, b in zip(host, (state, mean, t)))
    got = fl.abi_to_box(state.cpu().numpy()).astype(np.complex128)
    rel, mx = increment_errors(got, st, ref, st, p.K1)
    assert rel < INC_TOL["fp32"] and mx < INC_MAX_TOL["fp32"], (rel, mx)
    assert abs(mean.item() - mref) < 2e-5 * abs(mref)
    f.close()
