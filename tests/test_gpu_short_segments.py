"""The short segment lengths with more positions per CTA than the template ring holds, one spectrum
and a batch whose spectra start at odd unit numbers: every cell against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1711_10855_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(spec):
    return torch.from_numpy(spec.view(np.float32).copy()).cuda()


def _check(got, spec, zmax, zstep, m):
    ref = oracle.plane_rows(spec, zmax, zstep, m)
    err = np.max(np.abs(got.cpu().numpy().astype(np.float64) - ref), axis=1)
    assert np.all(err <= 1e-5 * np.max(ref, axis=1))   # NaN (an unwritten cell) fails


@pytest.mark.parametrize("n,zmax,zstep,L,m", [
    (400_004, 15, 1, 256, 32), (300_000, 10, 1, 256, 128), (400_004, 15, 1, 512, 60), (90_000, 0, 1, 512, 64),
    (250_000, 12, 1, 1024, 100), (120_004, 6, 1, 1024, 512), (300_000, 12, 1, 4096, 260), (300_000, 8, 1, 8192, 2048)])
def test_many_positions_per_cta(n, zmax, zstep, L, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_10855_gb300 import fdas
    spec = synth.noise_spectrum(n, seed=n + L)
    with fdas.Plan(n, zmax, zstep, L, m) as plan:
        plan.build_templates()
        out = torch.full((plan.n_z, n), float("nan"), dtype=torch.float32, device="cuda")
        plan.convolve_power(_dev(spec), out)
        plan.check()
        _check(out, spec, zmax, zstep, m)


@pytest.mark.parametrize("L,m", [(256, 64), (512, 64), (1024, 128)])
def test_batch_of_odd_unit_counts(L, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_10855_gb300 import fdas
    n, zmax = [4, 60_000, 452, 100_004, 8, 30_000, 200_000], [0, 5, 7, 3, 0, 1, 9]
    specs = [synth.noise_spectrum(k, seed=k) for k in n]
    with fdas.Batch(n, zmax, 1, L, m) as b:
        b.build_templates()
        planes = [torch.full((int(q), k), float("nan"), dtype=torch.float32, device="cuda") for q, k in zip(b.n_z, n)]
        b.convolve_power([_dev(s) for s in specs], planes, use_graph=L == 512)
        b.check()
        for spec, z, plane in zip(specs, zmax, planes):
            _check(plane, spec, z, 1, m)
