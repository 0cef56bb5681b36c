"""The inference kernel where an FP16 activation overflows: an infinite activation reaches the outputs
under its nine taps and no other, in either of the dilated layers.  Every block holds one bin whose first
channel overflows and one finite mark in the second channel, at each distance in turn that is one to
three dilation steps beyond the outermost taps; all weights from the first channel on are zero, so the
mark is the block's maximum wherever no tap reaches it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, K = 32, 9


def params(n_out, layer):
    """Channel 1 passes x through; channel 0 overflows FP16 at x = 64 in `layer` (1 or 2)."""
    W1, W2, W3 = np.zeros((C, 1, K)), np.zeros((C, C, K)), np.zeros((C, C, K))
    W1[0, 0, 4], W1[1, 0, 4] = (2000.0 if layer == 1 else 1.0), 1.0
    if layer == 2:
        W2[0, 0, 4] = 2000.0
    W2[1, 1, 4] = W3[1, 1, 4] = 1.0
    Wl = np.zeros((n_out, C))
    Wl[:, 1] = 1.0
    parts = [W1, np.zeros(C), W2, np.zeros(C), W3, np.zeros(C), Wl, np.arange(n_out)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


@pytest.mark.parametrize("window", [512, 768, 1024])
@pytest.mark.parametrize("layer,dilation", [(1, 4), (2, 16)])
def test_an_infinite_activation_stays_under_its_taps(window, layer, dilation):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_10855_gb300 import fdas
    hop, n_out = window // 2, 3
    beyond = [-7, -6, -5, 5, 6, 7]      # in dilation steps; the taps reach +-4
    blocks = len(beyond) * 64           # every residue of the position modulo 4 dilation steps (half of them at 512)
    A = np.ones(blocks * hop, dtype=np.complex64)
    for w in range(blocks):
        at = w * hop + 112 + w // len(beyond) % min(64, hop - 224)   # the marks stay inside the block
        A[at] = 10.0                                    # x = 64, the cap: 2000 x overflows
        A[at + dilation * beyond[w % len(beyond)]] = 6.5
    mark = 6.5 ** 2 * np.log(2.0)                       # the background's |A|^2 = 1 is the median
    with fdas.ZBand(window, n_out, 1) as net:
        net.set_params(params(n_out, layer))
        logits = torch.zeros((blocks, n_out), device="cuda")
        net.propose(torch.from_numpy(A.view(np.float32).copy()).cuda(), A.size, logits)
        net.check()
        got = logits.cpu().numpy()
    # one rounding to FP16 (the input's): 2^-11 relative
    assert np.all(np.abs(got - (mark + np.arange(n_out))) <= 2.0 ** -11 * mark + 1e-5)
