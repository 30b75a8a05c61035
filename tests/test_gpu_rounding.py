"""Rounding error of the FP32 transforms, seen through the nonlinear part of a
step and of an adjoint step (flat spectrum: every mode of the box the same
size), against the FP64 handle's on the same FP32 inputs.

Bars: the mean errors of the transforms of 2^n points that a step and an
adjoint step made before they ran on the alias-free grid, on these inputs
(two-line step, adjoint steps).  With the last pass's twiddles formed as FP32
products of two table entries, all three are exceeded (3.541e-7, 3.047e-7,
3.093e-7).
"""
import math

import numpy as np
import pytest
import torch

# (call, N1, N2): mean relative L2 error of the increment over SEEDS
BARS = {("step", 1024, 2048): 3.376e-7, ("adjoint", 2048, 1024): 3.040e-7, ("adjoint", 2048, 4096): 3.088e-7}
SEEDS = range(8)
T0 = 20.0


def _flat(f, seed, amp):
    """Every mode of the box of size amp, random phases, ABI layout."""
    rng = np.random.default_rng(seed)
    z = amp * np.exp(2j * np.pi * rng.random((f.K2 + 1, 2 * f.K1 + 1)))
    z[0, :f.K1] = np.conj(z[0, f.K1 + 1:][::-1])
    z[0, f.K1] = 0
    return torch.from_numpy(z).cuda().to(torch.complex64)


def _scalar(v):
    return torch.full((1,), v, dtype=torch.float64, device="cuda")


def mean_error(fl, call, n1, n2):
    errs = []
    for seed in SEEDS:
        # amplitudes over an octave: g and its row sums over two binades
        amp = 1e-4 * 2 ** (seed / len(SEEDS))
        flags = fl.FLAME_NONLINEAR_ONLY
        probe = fl.Flame(n1, n2, t0=T0, dt=1.0, prec="fp64", flags=flags)
        st = _flat(probe, seed, amp)
        d = st.to(torch.complex128)
        s = d.clone()
        probe.step(s, _scalar(0.0), _scalar(T0), 1)
        dt = 2.0 ** round(math.log2(0.5 * (d.norm() / (s - d).norm()).item()))  # an increment of half the state
        probe.close()
        out = []
        for prec in ("fp32", "fp64"):
            f = fl.Flame(n1, n2, t0=T0, dt=dt, prec=prec, flags=flags)
            x = st.to(f.cdtype)
            if call == "step":
                y = x.clone()
                f.step(y, _scalar(0.0), _scalar(T0), 1)
            else:
                x = _flat(f, 100 + seed, 1.0).to(f.cdtype)
                y = f.adjoint(st.to(f.cdtype), _scalar(0.0), _scalar(T0), 1, 1, x, _scalar(0.0))[0]
            out.append(y.to(torch.complex128) - x.to(torch.complex128))
            f.close()
        errs.append(((out[0] - out[1]).norm() / out[1].norm()).item())
    return float(np.mean(errs))


@pytest.mark.gpu
@pytest.mark.parametrize("call,n1,n2", list(BARS))
def test_increment_error_is_that_of_table_twiddles(fl, monkeypatch, call, n1, n2):
    monkeypatch.setenv("FLAME_FORCE_VARIANTS", "1,0")
    err = mean_error(fl, call, n1, n2)
    print(f"\n{call} {n1}x{n2}: {err:.4e}")
    assert err <= BARS[call, n1, n2]
