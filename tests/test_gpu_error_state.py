"""A refused call leaves no error behind for the calls after it."""
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["c128", "df64"])
def test_plans_work_after_a_refused_copy(qfdlib, prec):
    torch.cuda.empty_cache()
    short = torch.zeros(12 << 20, dtype=torch.uint8, device="cuda")  # a V or psi of 128^3 takes 16 or 32 MB
    torch.cuda.synchronize()
    with Q.Plan(128, 0.1, 1.3, 1e-3, 2, precision=prec) as p:
        assert p.lib.qfd_set_potential(p.h, short.data_ptr(), 1) == Q.ERR_CUDA  # the copy checks the range
        with Q.Plan(32, 0.1, 1.3, 1e-3, 2, precision=prec) as q:
            q.fill_potential("ho", (1.0,))
            q.fill_psi_uniform(0, 3)
            q.step(0, 2)
        p.fill_potential("ho", (1.0,))
        p.fill_psi_uniform(0, 3)
        p.step(0, 2)
        assert torch.isfinite(torch.from_numpy(p.get_psi(0)).abs()).all()
