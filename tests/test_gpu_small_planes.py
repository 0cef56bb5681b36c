"""Planes of few units at the segment lengths whose CTAs hold fewer segments then: one, two, four, ...
segments per CTA, ragged last groups, and CTAs with segments missing over many positions; every cell
against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1711_10855_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,m,n,zmax", [
    (1024, 256, 4, 0), (1024, 256, 768 * 3 + 4, 10), (1024, 256, 768 * 21, 14), (1024, 64, 960 * 37 + 8, 12),
    (1024, 512, 512 * 75, 7), (1024, 256, 768 * 17, 60),
    (4096, 1024, 4, 0), (4096, 1024, 3072 * 3 - 4, 20), (4096, 512, 3584 * 5, 25), (4096, 2048, 2048 * 13, 30),
    (4096, 1024, 3072 * 9, 80),
    (8192, 2048, 4, 0), (8192, 2048, 6144 * 3, 20), (8192, 1024, 7168 * 4 - 8, 30), (8192, 2048, 6144 * 5, 90)])
def test_plane_of_few_units(L, m, n, zmax):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_10855_gb300 import fdas
    spec = synth.noise_spectrum(n, seed=n + L)
    with fdas.Plan(n, zmax, 1, L, m) as plan:
        plan.build_templates()
        out = torch.full((plan.n_z, n), float("nan"), dtype=torch.float32, device="cuda")
        plan.convolve_power(torch.from_numpy(spec.view(np.float32).copy()).cuda(), out)
        plan.check()
    ref = oracle.plane_rows(spec, zmax, 1, m)
    err = np.max(np.abs(out.cpu().numpy().astype(np.float64) - ref), axis=1)
    assert np.all(err <= 1e-5 * np.max(ref, axis=1))   # NaN (an unwritten cell) fails
