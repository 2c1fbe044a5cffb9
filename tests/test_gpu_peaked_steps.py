"""One complex128 step of large lattices whose z lines take several warps, against
the stencil form of H_K(2).

4 sin^2(k / 2) is the symbol of the second difference, so on a periodic lattice
H_K(2) psi is (6 psi - the six neighbours) / (2 M A^2) exactly, formed here on the
device without a transform.

Tolerance: with V = 0 and dtau max T = 1 the transforms enter a step by half the
weight of psi' itself, and a step takes six of them.  A 64-bit transform is off by up
to 2e-16 (relative L2), so a step agrees to sqrt(6) 2e-16 = 5e-16, which also holds
the 1e-16 each of the update and of the stencil.
"""
import numpy as np
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
A, M = 0.1, 1.3
DT = 2 * A * A * M / 12
TOL = 5e-16


def step(n, psi):
    out = torch.empty_like(psi)
    with Q.Plan(n, A, M, DT, 2, ortho_every=1000) as p:
        p.fill_potential("zero")
        torch.cuda.synchronize()
        p.set_psi(0, psi)
        p.step(0, 1)
        p.get_psi(0, out)
        p.sync()
    return out


def reference(psi):
    s = -6.0 * psi
    for ax in range(3):
        for d in (1, -1):
            s += torch.roll(psi, d, ax)
    return psi + DT / (2 * M * A * A) * s


def rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


def state(n, kind):
    g = torch.Generator(device="cuda").manual_seed(n)

    def noise():
        return torch.view_as_complex(torch.rand(n, n, n, 2, generator=g, dtype=torch.float64, device="cuda") * 2 - 1)

    d = torch.arange(n, dtype=torch.float64, device="cuda") - n // 2
    if kind in ("site", "planes"):
        psi = torch.zeros(n, n, n, dtype=torch.complex128, device="cuda")
        if kind == "site":
            psi[n // 3, 1, n - 2] = 1.0 + 0.3j
        else:  # all-zero lines along two axes
            psi[0, 0] = noise()[0, 0]
        return psi
    psi = noise()
    if kind == "floor":  # a state of a few sites' width on a floor of noise
        e = torch.exp(-d ** 2 / 4.5)
        psi = 1e-9 * psi + (0.8 + 0.7j) * e[:, None, None] * e[None, :, None] * e[None, None, :]
    if kind == "decay":  # down to below 1e-290: threads of a line far below its largest element
        e = d.abs() / (n // 2)
        psi *= 10.0 ** (-290.0 * e[:, None, None] ** 4 - 30.0 * e[None, :, None] - 30.0 * e[None, None, :])
    return psi


@pytest.mark.parametrize("n,kind", [(192, "site"), (512, "noise"), (512, "site"), (512, "floor"), (512, "decay"),
                                    (512, "planes"), (1024, "site"), (1024, "floor")])
def test_step_matches_the_stencil(qfdlib, n, kind):
    psi = state(n, kind)
    got = step(n, psi)
    assert rel(got, reference(psi)) < TOL


def test_lines_outside_the_fixed_point_range_512(qfdlib):
    n = 512
    psi = state(n, "noise")
    ref = reference(psi)
    for k in (-965, 940):  # below and above the exponents that fixed point covers
        got = step(n, psi * 2.0 ** k)
        assert rel(got * 2.0 ** -k, ref) < TOL
    psi[3, 4, 5] = float("nan")
    assert not bool(torch.isfinite(torch.view_as_real(step(n, psi))).any())
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [8, 16, 32, 64, 128, 256, 512])
def test_lines_of_different_kinds_in_one_warp(qfdlib, n):
    # constant along y: of the z lines of a warp one holds all of the state, below the
    # fixed-point range, and the others are zero
    psi = state(n, "noise")[:, :1, :].expand(n, n, n).contiguous() * 2.0 ** -970
    assert rel(step(n, psi) * 2.0 ** 970, reference(psi * 2.0 ** 970)) < TOL
