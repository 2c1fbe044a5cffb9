"""Passes B, C and D of small lattices as one launch over planes (k_plane)
against the separate passes, which hand-set launch shapes select.

Both run the same line transforms; complex64 and complex128 kernels may differ
in where the compiler fuses a multiply-add, so they agree to rounding (the
bounds of tests/test_gpu_autotune.py), double-float bit for bit.
"""
import numpy as np
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu

POLICY = {"c128": 0, "c64": 1, "df64": 2}
TOL = {"df64": 0.0, "c128": 1e-14, "c64": 2e-6}


@pytest.mark.parametrize("prec,n", [(p, n) for p in POLICY for n in (8, 16, 32, 64, 96, 128) if n <= 32 or p == "c64"])
@pytest.mark.parametrize("kin", [2, 3])
def test_plane_pass_matches_the_separate_passes(qfdlib, prec, n, kin):
    res = []
    for shape in (None, (0, 0, 0)):
        with Q.Plan(n, 0.1, 1.3, 1e-4, kin, ortho_every=3, precision=prec) as p:
            if shape:
                p.set_tuning(POLICY[prec], *shape)
            p.fill_potential("cornell", (0.3, 0.2))
            p.fill_psi_uniform(0, 4)
            p.set_parity(0, -1)
            p.step(0, 4)
            e = p.energy(0)  # the Parseval instance, whose W the next step goes on from
            p.step(0, 3)
            res.append((p.get_psi(0), e))
    (a, ea), (b, eb) = res
    assert np.linalg.norm(a - b) <= TOL[prec] * np.linalg.norm(b)
    assert abs(ea[0] - eb[0]) <= max(TOL[prec], 1e-14) * abs(eb[0])
