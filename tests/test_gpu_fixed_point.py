"""The complex128 line transforms run on 64-bit integers scaled per line
(fft_line_fx in csrc/qfd_kernels.cuh); lines outside the range of exponents
they cover take the FP64 transform.

Tolerance: a step is six line transforms and the update.  numpy's transforms
are off by about 2e-16 sqrt(log2 n) each, the fixed-point ones by less, and the
transforms enter the update times dtau T <= 1, so one step agrees to 2e-15 in
relative L2; scaling psi by a power of two scales every exponent and nothing
else, so inside the covered range it gives the same bits.
"""
import numpy as np
import pytest

from oracle import qfd_oracle as O
from paper_2006_16935_gb300 import inputs
from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu

A, M, KIN = 0.1, 1.3, 2


def step(n, psi, V, steps=1, tuning=None):
    dt = 0.5 / O.kinetic_max(n, A, M, KIN, 0)
    with Q.Plan(n, A, M, dt, KIN, ortho_every=1000) as p:
        if tuning:
            p.set_tuning(0, *tuning)
        p.set_potential(V)
        p.set_psi(0, psi)
        p.step(0, steps)
        return p.get_psi(0)


def reference(n, psi, V):
    dt = 0.5 / O.kinetic_max(n, A, M, KIN, 0)
    T = O.kinetic_symbol(n, A, M, KIN)
    hk = np.fft.ifftn(T * np.fft.fftn(psi))
    h = 0.5 * dt * V
    return (1 - h) / (1 + h) * psi - dt / (1 + h) * hk


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def states(n, kind):
    psi = inputs.uniform_psi(n, 5)
    if kind == "delta":  # one site far above the rest: lines of every scale
        psi[n // 2, 1, n - 1] = 1e12
    if kind == "decay":  # 1 down to below 1e-280 along each axis (FP64 lines among them)
        d = np.abs(np.arange(n) - n // 2) / (n // 2)
        psi = psi * 10.0 ** (-290.0 * (d[:, None, None] ** 4) - 30.0 * d[None, :, None] - 30.0 * d[None, None, :])
    if kind == "planes":  # all-zero lines along two axes
        psi[1:] = 0.0
        psi[:, 1:] = 0.0
    if kind == "constant":  # the largest growth a transform can have
        psi = np.full((n, n, n), 1.0 - 2.0 ** -53, dtype=np.complex128) * (1 + 1j)
    return psi


@pytest.mark.parametrize("n", [8, 16, 32, 64, 96, 128, 192, 256])
@pytest.mark.parametrize("kind", ["noise", "delta", "decay", "planes", "constant"])
def test_one_step_matches_the_64_bit_transform(qfdlib, n, kind):
    V = O.potential(n, A, "cornell", (0.3, 0.2))
    psi = states(n, kind)
    assert rel(step(n, psi, V), reference(n, psi, V)) < 2e-15


@pytest.mark.parametrize("n", [16, 96, 256])
def test_scaling_by_powers_of_two(qfdlib, n):
    V = O.potential(n, A, "ho", (1.0,))
    psi = inputs.uniform_psi(n, 6)
    base = step(n, psi, V)
    for k in (-800, -3, 800):  # covered: the same bits
        assert np.array_equal(np.ldexp(step(n, np.ldexp(psi.view(float), k).view(complex), V).view(float), -k),
                              base.view(float))
    for k in (-965, 940):  # below and above: the FP64 transform
        got = np.ldexp(step(n, np.ldexp(psi.view(float), k).view(complex), V).view(float), -k).view(complex)
        assert rel(got, base) < 4e-15


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_sites_stay_non_finite(qfdlib, bad):
    n = 32
    psi = inputs.uniform_psi(n, 7)
    psi[3, 4, 5] = bad
    got = step(n, psi, np.zeros((n, n, n)))
    assert not np.isfinite(got).all(axis=0).any()


@pytest.mark.parametrize("n", [64, 192, 512])
def test_every_shape_gives_the_same_bits(qfdlib, n):
    # fixed point leaves nothing to contraction except the update in FP64
    V = O.potential(n, A, "cornell", (0.3, 0.2))
    psi = inputs.uniform_psi(n, 8)
    outs = [step(n, psi, V, 2, t) for t in [(0, -1, 0), (1, 0, 0), (0, 1, 1)]]
    for o in outs[1:]:
        assert rel(o, outs[0]) < 1e-15


def fdtd_reference(n, psi, V, dt):
    s = np.zeros_like(psi)
    for ax in range(3):
        lo = [slice(None)] * 3
        hi = [slice(None)] * 3
        lo[ax], hi[ax] = slice(0, n - 1), slice(1, n)
        s[tuple(hi)] += psi[tuple(lo)]
        s[tuple(lo)] += psi[tuple(hi)]
    h = 0.5 * dt * V
    return (1 - h) / (1 + h) * psi - dt / (1 + h) * (6 * psi - s) / (2 * M * A * A)


@pytest.mark.parametrize("n", [8, 96, 128])
@pytest.mark.parametrize("kind", ["noise", "delta", "decay", "planes"])
def test_stencil_sums_match_site_by_site(qfdlib, n, kind):
    # the neighbour sum on integers: within a few rounding errors of its largest
    # term at every site (also where the six span many scales, or are all zero)
    V = O.potential(n, A, "cornell", (0.3, 0.2), "offgrid")
    psi = states(n, kind)
    dt = 0.5 * 2 * M * A * A / 12
    with Q.Plan(n, A, M, dt, 0, ortho_every=1000, centre="offgrid") as p:
        p.set_potential(V)
        p.set_psi(0, psi)
        p.step(0, 1)
        got = p.get_psi(0)
    want = fdtd_reference(n, psi, V, dt)
    big = np.abs(psi)
    pad = np.pad(big, 1)
    for ax in range(3):
        for sh in (0, 2):
            w = [slice(1, n + 1)] * 3
            w[ax] = slice(sh, sh + n)
            big = np.maximum(big, pad[tuple(w)])
    assert np.all(np.abs(got - want) <= 16 * 2.0 ** -53 * big + 1e-300)
