"""qfd_set_psi / qfd_get_psi with device memory: lattices that the conversion kernels reach
in place, the ones that go through a copy, and buffers that end inside the lattice."""
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def plan(n, prec):
    p = Q.Plan(n, 0.1, 1.3, 1e-3, 2, precision=prec, ortho_every=10)
    p.fill_potential("ho", (1.0,))
    return p


def noise(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    return torch.view_as_complex(torch.rand(n, n, n, 2, generator=g, dtype=torch.float64, device="cuda") * 2 - 1)


@pytest.mark.parametrize("prec", ["c64", "df64"])
def test_a_buffer_that_ends_inside_the_lattice_is_refused(qfdlib, prec):
    torch.cuda.empty_cache()
    short = torch.zeros(12 << 20, dtype=torch.uint8, device="cuda")  # of 32 MB
    with plan(128, prec) as p:
        p.fill_psi_uniform(0, 3)
        want = p.get_psi(0)
        torch.cuda.synchronize()
        assert p.lib.qfd_set_psi(p.h, 0, short.data_ptr(), 1) != Q.OK
        assert p.lib.qfd_get_psi(p.h, 0, short.data_ptr(), 1) != Q.OK
        assert (p.get_psi(0) == want).all() and not bool(short.any())


@pytest.mark.parametrize("prec", ["c64", "df64"])
def test_unaligned_lattices_go_through_a_copy(qfdlib, prec):
    n = 32
    psi = noise(n)
    buf = torch.zeros(2 * n ** 3 + 1, dtype=torch.float64, device="cuda")
    with plan(n, prec) as p, plan(n, prec) as q:
        buf[1:] = torch.view_as_real(psi).reshape(-1)  # 8 bytes off a site
        torch.cuda.synchronize()
        p.set_psi(0, psi)
        assert q.lib.qfd_set_psi(q.h, 0, buf.data_ptr() + 8, 1) == Q.OK
        p.step(0, 3)
        q.step(0, 3)
        want = torch.from_numpy(p.get_psi(0))
        assert q.lib.qfd_get_psi(q.h, 0, buf.data_ptr() + 8, 1) == Q.OK
        got = torch.view_as_complex(buf[1:].clone().reshape(n, n, n, 2)).cpu()
    assert bool((got == want).all())


@pytest.mark.parametrize("prec", ["c64", "df64"])
def test_reading_a_state_between_steps_changes_nothing(qfdlib, prec):
    n = 32
    psi, out = noise(n), torch.empty(n, n, n, dtype=torch.complex128, device="cuda")
    with plan(n, prec) as p, plan(n, prec) as q:
        torch.cuda.synchronize()
        p.set_psi(0, psi)
        q.set_psi(0, psi)
        p.step(0, 6)
        q.step(0, 3)
        q.get_psi(0, out)
        q.step(0, 3)
        assert (p.get_psi(0) == q.get_psi(0)).all()
