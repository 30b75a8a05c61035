"""CPU model of the step's transforms of 3 * 2^A points (csrc/line3.cuh) and
of the row pass built on them (csrc/flame_step.cuh): the per-thread indices,
paddings and twiddles of the kernels in NumPy.  Checks that every plan is the
DFT, that no exchange leaves its buffer or stores two points in one slot, and
that the folded half-length transforms and the post-processing give the
retained coefficients of |w|^2 on the alias-free grid and on a larger one."""
import math

import numpy as np
import pytest

PLANS = [(a, f) for f, lo in ((1, 2), (2, 3), (4, 4)) for a in range(lo, 11)]
WAVES = (8, 16, 32)  # slots per shared-memory wavefront: two FP32 lines, one FP64, one FP32


class Plan:
    def __init__(self, a, f):
        lf = {1: 0, 2: 1, 4: 2}[f]
        self.L, self.ES, self.EP = 3 << a, 3 * f, 4 * f
        nb, mb = a - lf, lf + 2
        self.NQ = -(-nb // mb)
        self.q = [1 << (nb // self.NQ + (1 if i < nb % self.NQ else 0)) for i in range(self.NQ)]

    def radices(self, inv):
        return [self.ES] + self.q if inv else self.q + [self.ES]

    def pad(self, inv, s, w):
        r = self.radices(inv)
        ns = math.prod(r[:s])
        if s == 0:
            return math.lcm(r[0], w), 1
        return ns * r[s], (ns - ns * r[s]) % w

    def slots(self, w):
        m = self.L
        for inv in (True, False):
            for s in range(self.NQ):
                d, p = self.pad(inv, s, w)
                m = max(m, self.L + p * ((self.L - 1) // d))
        return (m + 7) & ~7

    def run(self, x, inv, w):
        """The transform of x by the kernels' passes, through the padded buffer."""
        r, L = self.radices(inv), self.L
        buf = np.full(self.slots(w), np.nan + 0j)
        regs, ns = None, 1
        for s, rad in enumerate(r):
            spectral = s == 0 if inv else s == self.NQ
            e = self.ES if spectral else self.EP
            T, B = L // e, e // rad
            t = np.arange(T)
            if s == 0:
                regs = x[t[:, None] + T * np.arange(e)[None, :]]
            else:
                d, p = self.pad(inv, s - 1, w)
                i = t[:, None] + T * np.arange(e)[None, :]
                if T % d == 0:
                    slot = (t + p * (t // d))[:, None] + (T + p * (T // d)) * np.arange(e)
                elif d % T == 0:
                    slot = i + p * (np.arange(e) * T // d)
                else:
                    slot = i + p * (i // d)
                assert np.array_equal(slot, i + p * (i // d))
                regs = buf[slot]
            out = np.empty_like(regs)
            dft = np.exp((2j if inv else -2j) * np.pi * np.outer(np.arange(rad), np.arange(rad)) / rad)
            for b in range(B):
                y = regs[:, b + B * np.arange(rad)]
                m = (t + b * T) % ns
                y = y * np.exp((2j if inv else -2j) * np.pi * np.outer(m, np.arange(rad)) / (rad * ns))
                out[:, b + B * np.arange(rad)] = y @ dft.T
            if s == len(r) - 1:
                res = np.empty(L, dtype=complex)
                res[t[:, None] + T * np.arange(e)[None, :]] = out
                return res
            d, p = self.pad(inv, s, w)
            buf[:] = np.nan
            for b in range(B):
                j = t + b * T
                base = rad * j + p * (j // (d // rad)) if s == 0 else (j // ns) * (ns * rad + p) + j % ns
                for q in range(rad):
                    slot = base + q * ns
                    assert slot.min() >= 0 and slot.max() < len(buf)
                    assert np.all(np.isnan(buf[slot]))
                    buf[slot] = out[:, b + B * q]
            assert np.count_nonzero(~np.isnan(buf)) == L
            ns *= rad


@pytest.mark.parametrize("a,f", PLANS)
def test_plan_is_the_dft_in_its_buffer(a, f):
    pl = Plan(a, f)
    assert math.prod(pl.radices(True)) == pl.L and pl.L % pl.EP == 0
    rng = np.random.default_rng(a * 8 + f)
    x = rng.standard_normal(pl.L) + 1j * rng.standard_normal(pl.L)
    for w in WAVES:
        np.testing.assert_allclose(pl.run(x, True, w), np.fft.ifft(x) * pl.L, atol=1e-9)
        np.testing.assert_allclose(pl.run(x, False, w), np.fft.fft(x), atol=1e-9)


@pytest.mark.parametrize("a,K", [(2, 7), (2, 3), (3, 15), (4, 31), (4, 25), (6, 127), (6, 100)])
def test_row_pass_keeps_the_retained_harmonics_alias_free(a, K):
    # rows of 2 L points, L = 3 * 2^a, harmonics |k| <= K: even points from
    # W[n] + W[n - L], odd ones from (W[n] - W[n - L]) exp(2 pi i n / 2L), then
    # the real transform of |w|^2, against a transform of 4K + 1 points or more
    L = 3 << a
    assert 2 * L >= 3 * K + 1
    rng = np.random.default_rng(K)
    W = {k: complex(*rng.standard_normal(2)) for k in range(-K, K + 1)}
    n = np.arange(L)
    up = np.array([W.get(int(i), 0) for i in n])
    um = np.array([W.get(int(i) - L, 0) for i in n])
    w = np.exp(2j * np.pi * n / (2 * L))
    pl = Plan(a, 1)
    even, odd = pl.run(up + um, True, 8), pl.run((up - um) * w, True, 8)
    H = pl.run(np.abs(even) ** 2 + 1j * np.abs(odd) ** 2, False, 8)
    G = np.full(K + 1, np.nan + 0j)
    for k in range(L // 2 + 1):
        h, hc = H[k], np.conj(H[(L - k) % L])
        E, O = (h + hc) / 2, (h - hc) / 2j
        if k <= K:
            G[k] = E + O * np.conj(w[k])
        if 0 < L - k <= K:
            G[L - k] = np.conj(E - O * np.conj(w[k]))
    N = 8 * (K + 1)
    full = np.zeros(N, dtype=complex)
    for k, v in W.items():
        full[k % N] = v
    ref = np.fft.fft(np.abs(np.fft.ifft(full) * N) ** 2)[: K + 1] / N
    np.testing.assert_allclose(G / (2 * L), ref, atol=1e-12 * np.abs(ref).max())
