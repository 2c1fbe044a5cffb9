"""complex64 at 1024^3: the x transforms of pass A, the cadence and the energy
run on 16-column tiles with schedule 2 (radix 16, 16, 4; Shape::XR in
csrc/qfd_kernels.cuh).  Checked against the complex128 plan, and against the
8-column tiles, through a projection and an energy check.

Bound: FP32 transforms round at about eps32 log2(n) each (2e-6 for ten steps in
tests/test_gpu_parity.py); two steps and a projection stay within it.
"""
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu


def run(prec, shape=None):
    import torch

    n = 1024
    out = torch.empty(n, n, n, dtype=torch.complex128, device="cuda")
    with Q.Plan(n, 0.05, 1.0, 2e-4, 2, ortho_every=2, precision=prec) as p:
        if shape:
            p.set_tuning(1, *shape)
        p.fill_potential("softcoul", (0.01,))
        p.fill_psi_uniform(0, 9)
        p.set_parity(0, 1)
        p.step(0, 2)
        e = p.energy(0)
        p.step(0, 1)
        p.get_psi(0, out)
    return out, e


def test_cadence_on_wide_tiles_matches_complex128(qfdlib):
    torch = pytest.importorskip("torch")
    ref, er = run("c128")
    for shape in (None, (0, -1, 1)):
        got, e = run("c64", shape)
        got -= ref
        assert float(torch.linalg.vector_norm(got)) <= 2e-6 * float(torch.linalg.vector_norm(ref))
        assert abs(e[0] - er[0]) <= 1e-6 * abs(er[0])
        del got
        torch.cuda.empty_cache()
