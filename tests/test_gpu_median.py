"""The median behind the proposal's input scale, where its counters could overflow or its digits meet:
more values per thread than a byte counts, one value throughout, values around a binade's edge,
an odd start, non-finite values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _spectrum(kind, n):
    rng = np.random.default_rng(n)
    if kind == "one-value":
        return np.full(n, 3.0, dtype=np.complex64)
    if kind == "binade-edge":
        return np.sqrt(rng.choice(np.float32([0.99999994, 1.0, 1.0000001, 1e-40, 4e37]), n)).astype(np.complex64)
    if kind == "non-finite":
        s = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
        s[::7] = np.inf
        s[::11] = -np.nan
        return s
    return (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)


@pytest.mark.parametrize("kind,n,shift", [
    ("noise", 1, 0), ("noise", 2, 1), ("noise", 2047, 1), ("noise", 2048, 0), ("noise", 100_003, 1),
    ("one-value", 5_000_001, 0), ("binade-edge", 300_001, 1), ("non-finite", 60_000, 0), ("noise", 40_000_000, 1)])
def test_scale_is_the_exact_median(kind, n, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_10855_gb300 import fdas
    spec = _spectrum(kind, n)
    buf = torch.empty(n + shift, dtype=torch.complex64, device="cuda")
    buf[shift:] = torch.from_numpy(spec)
    d = torch.view_as_real(buf)[shift:]          # 8-byte aligned when shift is 1
    out = torch.empty((1, 1024), dtype=torch.float32, device="cuda")
    for _ in range(2):
        fdas.zband_spectrum_windows(d, n, 1024, 512, out, 1)
    a = d.cpu().numpy()
    # |A|^2 as the kernel rounds it: fma(re, re, im * im)
    p = (a[:, 0].astype(np.float64) ** 2 + (a[:, 1] * a[:, 1]).astype(np.float64)).astype(np.float32)
    med = np.sort(p)[(n - 1) // 2]               # NaN last, as its bits order
    scale = np.float32(np.log(2.0)) / med if med > 0 else np.float32(0)
    k = min(n, 768)
    with np.errstate(invalid="ignore"):
        want = np.fmin(p[:k] * scale, np.float32(64))
    got = out.cpu().numpy()[0]
    np.testing.assert_allclose(got[256:256 + k], want, rtol=3e-7)
    assert not got[:256].any() and not got[256 + k:].any()
