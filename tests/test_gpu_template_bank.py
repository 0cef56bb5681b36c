"""The template bank at the edges of its build: no acceleration at all, more panels than the
segment has points, the tap-by-tap quadrature of very large zmax, the longest segment."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zmax,zstep,L,m", [
    (0, 1, 256, 4), (0, 1, 8192, 4096), (30, 3, 256, 128), (6000, 3000, 256, 8), (1638, 546, 8192, 4096),
    (60000, 30000, 8192, 4096), (120000, 60000, 512, 16)])
def test_bank_at_the_edges(zmax, zstep, L, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_10855_gb300 import fdas
    with fdas.Plan(4096, zmax, zstep, L, m) as plan:
        plan.build_templates()
        for zi in {0, plan.n_z // 2, plan.n_z - 1, plan.n_z // 4}:
            z = -zmax + zi * zstep
            got, ref = plan.template_taps(zi), oracle.template(z, m)
            # a sample's phase is pi times a product of size |z| rounded to 2^-53 a few times; the taps
            # are divided by the raw norm
            norm = np.linalg.norm(oracle.template(z, m, normalise=False))
            assert np.max(np.abs(got - ref)) <= 1e-12 + 8 * np.pi * abs(z) * 2.0 ** -53 / norm, z
            want = oracle.template_spectrum(z, m, L)
            spec = plan.template_spectrum(zi).astype(np.complex128)
            # complex64 rounding of each part, and the taps' error summed over m + 1 taps
            bound = 2.0 ** -23 * np.max(np.abs(want)) + (m + 1) * np.max(np.abs(got - ref)) / L
            assert np.max(np.abs(spec - want)) <= bound, z
