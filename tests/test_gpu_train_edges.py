"""Training and windowed inference where the register tiles end inside a window: the narrowest
window, widths whose layers are no whole number of tiles, one window, and targets of all kinds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import zband as oz
    from paper_1711_10855_gb300 import fdas
    from test_gpu_zband import NAMES, FP32_MODEL, chirp_spectrum, dev, make_params, unflat


@pytest.mark.parametrize("W,Z,B", [(384, 5, 1), (512, 33, 7), (640, 21, 3), (1024, 201, 2), (2048, 9, 2)])
def test_train_step_at_tile_edges(W, Z, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    vec, p64 = make_params(Z, 61)
    x = oz.windows(oz.power_x(chirp_spectrum(8192, 62)), W, W // 2, B).astype(np.float32)
    tgt = (np.random.default_rng(63).random((B, Z)) < 0.2).astype(np.float32)
    with fdas.ZBand(W, Z, B + 2) as net:
        net.set_params(vec)
        logits = torch.empty((B, Z), dtype=torch.float32, device="cuda")
        # an input that starts 4 bytes off a 16-byte boundary
        flat = torch.empty(B * W + 1, dtype=torch.float32, device="cuda")
        xd = flat[1:].view(B, W)
        xd.copy_(torch.from_numpy(x))
        net.predict(xd, B, logits, half_weights=False)
        got_l = logits.cpu().numpy()
        loss = net.train_step(xd, dev(tgt), B, 1e-3)
        g = unflat(net.gradients(), Z)
    want_l, bound_l = oz.logits_error_bound(p64, x.astype(np.float64), **FP32_MODEL)
    assert np.all(np.abs(got_l - want_l) <= bound_l)
    loss_o, _ = oz.loss_and_grads(p64, x.astype(np.float64), tgt.astype(np.float64))
    assert abs(loss - loss_o) <= 1e-5 * max(1.0, abs(loss_o))
    g_o, bnd = oz.grads_error_bound(p64, x.astype(np.float64), tgt.astype(np.float64))
    for k in NAMES:
        err = np.abs(g[k] - g_o[k])
        assert np.all(err <= bnd[k]), (k, float(np.max(err / np.maximum(bnd[k], 1e-300))))
