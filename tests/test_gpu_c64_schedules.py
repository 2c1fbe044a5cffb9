"""The radix schedules of complex64 transforms are equally exact: one step with the
two-stage y pass (the default from n = 256 on) and z pass against the stencil form of
H_K(2) on a periodic lattice, next to the radix-8 schedule.

Tolerance: both schedules round every output of a stage once, the two-stage one in fewer
stages; its twiddles, products of at most four rounded values, add about what that saves.
10% is left for the different roundings of one state.
"""
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
A, M = 0.1, 1.3
DT = 2 * A * A * M / 12


def step(n, psi, tuning):
    out = torch.empty_like(psi)
    with Q.Plan(n, A, M, DT, 2, precision="c64", ortho_every=1000) as p:
        if tuning:
            p.set_tuning(1, *tuning)
        p.fill_potential("zero")
        torch.cuda.synchronize()
        p.set_psi(0, psi)
        p.step(0, 1)
        p.get_psi(0, out)
        p.sync()
    return out


@pytest.mark.parametrize("n", [128, 256, 512, 1024])
def test_two_stage_schedules_are_as_exact_as_radix_8(qfdlib, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.view_as_complex(torch.rand(n, n, n, 2, generator=g, device="cuda") * 2 - 1).to(torch.complex128)
    ref = -6.0 * psi
    for ax in range(3):
        for d in (1, -1):
            ref += torch.roll(psi, d, ax)
    ref = psi + DT / (2 * M * A * A) * ref
    norm = torch.linalg.vector_norm(ref)

    def err(tuning):
        return float(torch.linalg.vector_norm(step(n, psi, tuning) - ref) / norm)

    radix8 = err((0, -1, 0))
    for tuning in (None, (2, -1, 0), (2, 2, 0)):
        assert err(tuning) < 1.1 * radix8, tuning
    torch.cuda.empty_cache()
