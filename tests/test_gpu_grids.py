"""Truncations at which the alias-free grid's lines of 3 * 2^a points change
length (3 K + 1 just below and just above it), and transform sizes at which
the 2-D transforms change kernels, through the C ABI against the oracle.

Bars: the increment bars of increments.py for a step, those of
test_gpu_adjoint.py for a gradient, those of test_gpu_fft.py for a transform.
"""
import dataclasses

import numpy as np
import pytest
import torch

from conftest import rel_l2
from increments import INC_MAX_TOL, INC_TOL, dt_for_fraction, increment_errors
from paper_0911_2889_gb300 import inputs

# (N1, N2, K1, K2): 3 K + 1 <= 48, 96, 192, 384, or one harmonic more
BOXES = [(16, 32, 1, 7), (16, 64, 3, 15), (64, 128, 15, 16), (128, 64, 31, 15), (256, 128, 32, 31), (128, 256, 16, 32),
         (256, 256, 63, 63), (512, 256, 64, 5), (64, 1024, 15, 255), (512, 1024, 127, 128)]
FFT_SHAPES = [(32, 64), (32, 1024), (512, 64), (512, 512), (1024, 512), (1024, 1024), (2048, 2048), (4096, 64), (64, 8192),
              (4096, 1024)]
FFT_TOL = {"fp64": 1e-13, "fp32": 3e-6}


def _host(fl, t):
    return fl.abi_to_box(t.cpu().numpy()).astype(np.complex128)


def _scalar(x):
    return torch.full((1,), float(x), dtype=torch.float64, device="cuda")


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("box", BOXES)
def test_step_increment_at_line_lengths(fl, orc, prec, box):
    n1, n2, K1, K2 = box
    p = orc.Params(n1, n2, K1=K1, K2=K2, t0=20.0, flags=fl.FLAME_NONLINEAR_ONLY)
    st = inputs.flat_ic(n1, n2, 13, 1e-3, K1=K1, K2=K2)
    if prec == "fp32":
        st = st.astype(np.complex64).astype(np.complex128)
    p = dataclasses.replace(p, dt=dt_for_fraction(orc, p, st, 0.0, 0.5))
    ref, _, _ = orc.step(p, st, 0.0, p.t0, 1)
    f = fl.Flame(n1, n2, K1=K1, K2=K2, prec=prec, gamma=p.gamma, t0=p.t0, dt=p.dt, flags=p.flags)
    state, mean, t = torch.from_numpy(fl.box_to_abi(st)).cuda().to(f.cdtype), _scalar(0.0), _scalar(p.t0)
    f.step(state, mean, t)
    rel, mx = increment_errors(_host(fl, state), st, ref, st, K1)
    assert rel < INC_TOL[prec] and mx < INC_MAX_TOL[prec], (rel, mx)
    f.close()


@pytest.mark.gpu
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
@pytest.mark.parametrize("box", BOXES[1:5] + BOXES[7:8])
def test_gradient_at_line_lengths(fl, orc, prec, tol, box):
    n1, n2, K1, K2 = box
    f = fl.Flame(n1, n2, K1=K1, K2=K2, prec=prec, t0=5.0, dt=0.05, gamma=0.8)
    st = inputs.spectrum_ic(n1, n2, min(8, K1, K2), seed=5, amp=0.1, K1=K1, K2=K2)
    st0 = torch.from_numpy(fl.box_to_abi(st)).cuda().to(f.cdtype)
    mean0, t0 = _scalar(0.1), _scalar(5.0)
    s, m, t = st0.clone(), mean0.clone(), t0.clone()
    f.step(s, m, t, 3)
    _, lam, lam0 = f.area(s, m, t, grad=True)
    g, gm, gg = f.adjoint(st0, mean0, t0, 3, 2, lam, lam0)
    p = orc.Params(n1, n2, K1=K1, K2=K2, t0=5.0, dt=0.05, gamma=0.8)
    _, gr, ggr = orc.area_grad(p, _host(fl, st0), 0.1, 5.0, 3)
    gr0 = gr.copy()
    gr0[K1, 0] = 0
    assert rel_l2(_host(fl, g), gr0) < tol
    assert abs(gm.item() - gr[K1, 0].real) <= tol * abs(gr[K1, 0].real)
    assert abs(gg.item() - ggr) <= tol * max(abs(ggr), 1e-12)
    f.close()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", FFT_SHAPES)
def test_transforms_at_kernel_changes(fl, orc, prec, shape):
    n1, n2 = shape
    f = fl.Flame(n1, n2, prec=prec)
    x = torch.from_numpy(inputs.real_field(n1, n2, seed=n1 + n2)).cuda().to(f.rdtype)
    X = f.fft_r2c(x)
    ref = orc.rfft2(x.double().cpu().numpy())
    assert rel_l2(X.cpu().numpy(), ref) < FFT_TOL[prec]
    Y = torch.from_numpy(ref).to(f.cdtype).cuda()
    y = f.fft_c2r(Y)
    assert rel_l2(y.cpu().numpy(), orc.irfft2(Y.cpu().numpy().astype(np.complex128), n2)) < FFT_TOL[prec]
    f.close()
