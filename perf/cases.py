"""Timed cases: the work that a program using this library has it do, through the public calls of
paper_1711_10855_gb300.fdas.  Sizes are those of the library's workloads and tests, or of the same
kind: spectra of 2^16 to 2^22 bins, template lengths of an eighth to a half of the segment.

kinds of case
  plane   one spectrum, one plan that the program keeps: fdas.Plan.convolve_power
  fresh   a program that searches one spectrum: plan, template bank, plane, check
  batch   uneven de-dispersion trials in one call: fdas.Batch.convolve_power as a CUDA graph
  propose the z-band network over a whole spectrum: fdas.ZBand.propose
  pairs   the proposal's second half: logits -> (segment, template) list -> partial plane, without a
          host synchronisation (what ProposalSearch.search_async runs after the network)
  train   one optimiser step of the z-band network on a mini-batch

The tensor-core variant of the correlation (convolve_power_tc) is not listed: it is slower and less
accurate than the plain path on the same inputs, so a program has no reason to call it.
"""
import math

import numpy as np
import torch

from paper_1711_10855_gb300 import fdas, zband

DEV = "cuda"


# ----------------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------------
def _plane(name, n, zmax, zstep, L, m):
    return {"name": name, "kind": "plane", "n": n, "zmax": zmax, "zstep": zstep, "L": L, "m": m}


def listed():
    return [
        # the small workload (2^16 bins, z in [-20, 20], 64 taps): a quick look, latency counts
        _plane("small-512", 1 << 16, 20, 2, 512, 64),
        # a narrow acceleration range with the shortest segment: a million ragged bins, unit z step
        _plane("narrow-256", 1_000_004, 8, 1, 256, 32),
        # the spectra that label training windows (2^17 bins, the survey's templates): an ordinary call
        _plane("label-2048", 1 << 17, 200, 2, 2048, 512),
        # half the survey's acceleration range, templates half as long, ragged length
        _plane("mid-1024", 3_000_004, 100, 2, 1024, 256),
        # the survey plane: 2^22 bins, z in [-200, 200]
        _plane("survey-2048", 1 << 22, 200, 2, 2048, 512),
        # wide acceleration ranges need long templates, and those long segments
        _plane("wide-4096", 1 << 21, 400, 2, 4096, 1024),
        _plane("wider-8192", 1_500_012, 800, 4, 8192, 2048),
        # de-dispersion trials of uneven length, zmax 100 or 200 each, one launch
        {"name": "batch-2048", "kind": "batch", "count": 24, "lo": 1 << 18, "hi": 1 << 20, "L": 2048, "m": 512},
        # one spectrum searched by a program that starts from nothing
        {"name": "fresh-2048", "kind": "fresh", "n": 1 << 20, "zmax": 200, "zstep": 2, "L": 2048, "m": 512},
        # the proposal path on a survey spectrum, in its two halves
        {"name": "propose-survey", "kind": "propose", "n": 1 << 22, "Z": 201},
        {"name": "pairs-survey", "kind": "pairs", "n": 1 << 22, "zmax": 200, "zstep": 2, "signals": 0.3},
        # training: 256 windows of 1024 bins, 201 templates
        {"name": "train-256", "kind": "train", "batch": 256, "Z": 201},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bins(rng, lo, hi):
    n = _log_int(rng, lo, hi)
    return max(4, n - n % 4 + (4 if rng.random() < 0.3 else 0))


def draw(rng):
    kind = rng.choice(["plane", "plane", "plane", "plane", "fresh", "batch", "propose", "pairs", "train"])
    if kind in ("plane", "fresh"):
        # one-off searches use the short segments; the longest segments are for templates up to 2048 taps
        L = rng.choice([256, 512, 1024, 2048, 4096, 8192] if kind == "plane" else [512, 1024, 2048])
        m = int(L * rng.choice([0.125, 0.25, 0.25, 0.375, 0.5])) - 4 * rng.randrange(3)
        m = min(m, 2048)
        # a template spans about zmax bins: up to about 0.4 of the taps; up to about 400 templates
        zmax = m * rng.uniform(0.15, 0.4)
        zstep = rng.choice([s for s in (1, 2, 2, 4) if zmax / s <= 200] or [4])
        zmax = max(zstep, int(zmax) // zstep * zstep)
        Z = 2 * (zmax // zstep) + 1
        most = (8e8 if kind == "plane" else 2e8) / Z
        n = _bins(rng, 1 << 14, min(1 << 22, most))
        return {"kind": kind, "n": n, "zmax": zmax, "zstep": zstep, "L": L, "m": m}
    if kind == "batch":
        L, m = rng.choice([(512, 128), (1024, 256), (2048, 512), (2048, 512)])
        hi = _log_int(rng, 1 << 18, 1 << 20)
        return {"kind": "batch", "count": rng.randrange(3, 25), "lo": hi // 4, "hi": hi, "L": L, "m": m}
    if kind == "propose":
        return {"kind": "propose", "n": _bins(rng, 1 << 16, 1 << 22), "Z": rng.choice([101, 201, 201])}
    if kind == "pairs":
        return {"kind": "pairs", "n": _bins(rng, 1 << 18, 1 << 22), "zmax": rng.choice([100, 200]), "zstep": 2,
                "signals": round(rng.uniform(0.05, 0.5), 2)}
    return {"kind": "train", "batch": rng.choice([32, 64, 100, 128, 250, 256]), "Z": rng.choice([101, 201, 301])}


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
def _spectrum(n, zmax, seed, every=1 << 16):
    """rfft of unit noise with a constant-drift chirp per 2^16 bins (at least one), 3 to 15 sigma: a
    de-dispersed series' spectrum; (n, 2) float32."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    N = 2 * n
    x = torch.randn(N, generator=g, device=DEV, dtype=torch.float64)
    u = torch.arange(N, device=DEV, dtype=torch.float64) / N
    for _ in range(min(16, max(1, n // every))):
        z = rng.uniform(-0.9 * zmax, 0.9 * zmax)
        r0 = rng.uniform(0.02, 0.98) * n - 0.5 * z
        amp = 2 * rng.uniform(5.0, 30.0) / math.sqrt(N)
        x += amp * torch.cos(2 * math.pi * (r0 * u + 0.5 * z * u * u) + rng.uniform(0, 2 * math.pi))
    return torch.view_as_real(torch.fft.rfft(x)[:n].to(torch.complex64)).contiguous()


def _batch_sizes(case, seed):
    # the sizes belong to the case, not to the inputs: a plan is made for them
    rng = np.random.default_rng(case["hi"] + case["count"])
    n = (np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"])).astype(np.int64) // 4) * 4
    top = 200 if case["m"] >= 512 else case["m"] * 3 // 16 * 2
    return n, rng.choice([top // 4 * 2, top], case["count"]).astype(np.int32)


def _params(Z, seed):
    p = zband.init_params(Z, seed=seed % 1000).astype(np.float64)
    rng = np.random.default_rng(seed)
    C, K = 32, 9
    at = C * K
    for width in (C, C, C):   # a trained network's biases are not zero
        p[at:at + width] = rng.uniform(-0.1, 0.1, width)
        at += width + C * C * K
    return p.astype(np.float32)


def _power_x(spec):
    """min(|A|^2 ln 2 / lower median, 64), 64 bits."""
    p = spec.double().square().sum(-1)
    return (p * (math.log(2.0) / p.kthvalue((p.numel() + 1) // 2).values)).clamp(max=64.0)


def _logits(case, seed):
    """What a trained network gives: blocks without a signal low, blocks with one a band around +-z."""
    rng = np.random.default_rng(seed)
    zs = np.arange(-case["zmax"], case["zmax"] + 1, case["zstep"])
    nb = -(-case["n"] // zband.HOP)
    out = rng.normal(-7.0, 1.0, (nb, zs.size))
    on = rng.random(nb) < case["signals"]
    z = rng.uniform(0, case["zmax"], nb)
    d = np.minimum(np.abs(zs[None] - z[:, None]), np.abs(zs[None] + z[:, None]))
    out += on[:, None] * 11.0 * np.exp(-0.5 * (d / rng.uniform(3, 15, (nb, 1))) ** 2)
    return torch.from_numpy(out.astype(np.float32)).to(DEV)


def _windows(case, seed):
    B, Z = case["batch"], case["Z"]
    W, H = zband.WINDOW, zband.HOP
    rng = np.random.default_rng(seed)
    zs = np.linspace(-200, 200, Z)
    x = _power_x(_spectrum(B * H, 200, seed, every=1 << 13))
    win = torch.nn.functional.pad(x, (W // 4, W)).unfold(0, W, H)[:B].float().contiguous()
    lab = zband.band_masks(rng.uniform(-200, 200, B), zs, zband.HALF_BAND) * (rng.random(B) < 0.5)[:, None]
    return win, torch.from_numpy(lab.astype(np.float32)).to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("plane", "fresh"):
        geo = (case["n"], case["zmax"], case["zstep"], case["L"], case["m"])
        Z = 2 * (case["zmax"] // case["zstep"]) + 1
        s = {"kind": kind, "geo": geo, "spec": _spectrum(case["n"], case["zmax"], seed),
             "plane": torch.zeros((Z, case["n"]), device=DEV)}
        if kind == "plane":
            s["plan"] = fdas.Plan(*geo)
            s["plan"].build_templates()
        return s
    if kind == "batch":
        n, zmax = _batch_sizes(case, seed)
        b = fdas.Batch(n, zmax, 2, case["L"], case["m"])
        b.build_templates()
        specs = [_spectrum(int(k), int(z), seed + 7 * i) for i, (k, z) in enumerate(zip(n, zmax))]
        planes = [torch.zeros((int(q), int(k)), device=DEV) for q, k in zip(b.n_z, n)]
        return {"kind": kind, "batch": b, "specs": specs, "planes": planes}
    if kind == "propose":
        net = fdas.ZBand(zband.WINDOW, case["Z"], 1)
        net.set_params(_params(case["Z"], seed))
        return {"kind": kind, "net": net, "n": case["n"], "spec": _spectrum(case["n"], 200, seed),
                "logits": torch.zeros((net.n_blocks(case["n"]), case["Z"]), device=DEV)}
    if kind == "pairs":
        plan = fdas.Plan(case["n"], case["zmax"], case["zstep"], 2048, 512)
        plan.build_templates()
        cap = plan.n_seg * plan.n_z
        return {"kind": kind, "plan": plan, "spec": _spectrum(case["n"], case["zmax"], seed),
                "logits": _logits(case, seed), "pairs": torch.zeros(cap, dtype=torch.int32, device=DEV),
                "scratch": torch.zeros(fdas.zband_work_units_scratch_bytes(plan.n_seg, plan.n_z), dtype=torch.uint8,
                                       device=DEV),
                "plane": torch.zeros((plan.n_z, case["n"]), device=DEV)}
    net = fdas.ZBand(zband.WINDOW, case["Z"], case["batch"])
    net.set_params(_params(case["Z"], seed))
    win, lab = _windows(case, seed)
    return {"kind": kind, "net": net, "win": win, "lab": lab}


# ----------------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------------
HALO, THRESHOLD, REACH = 8, 0.1, 0.5   # the calibrated operating point of the proposal search


def run(s):
    kind = s["kind"]
    if kind == "plane":
        s["plan"].convolve_power(s["spec"], s["plane"])
        return s["plane"]
    if kind == "fresh":
        with fdas.Plan(*s["geo"]) as plan:
            plan.build_templates()
            plan.convolve_power(s["spec"], s["plane"])
            plan.check()
        return s["plane"]
    if kind == "batch":
        s["batch"].convolve_power(s["specs"], s["planes"], use_graph=True)
        return s["planes"]
    if kind == "propose":
        s["net"].propose(s["spec"], s["n"], s["logits"])
        return s["logits"]
    if kind == "pairs":
        plan, lg = s["plan"], s["logits"]
        fdas.zband_work_pairs(lg, lg.shape[0], plan.n_z, THRESHOLD, HALO, zband.HOP, plan.valid, plan.tmpl_len // 2,
                              plan.n_seg, s["pairs"], s["scratch"], host_count=False, reach_threshold=REACH)
        plan.convolve_power_pairs_device_count(s["spec"], s["plane"], s["pairs"],
                                               fdas.zband_work_units_count_ptr(s["scratch"], plan.n_seg),
                                               s["pairs"].numel())
        return {"pairs": s["pairs"], "plane": s["plane"]}
    net = s["net"]
    loss = net.train_step(s["win"], s["lab"], s["win"].shape[0], 1e-3)
    return {"loss": loss, "grads": net.gradients(), "params": net.get_params()}


# ----------------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------------
def _plane_work(n, Z, L, m, share=1.0):
    V = L - m
    nseg = -(-n // V)
    lg = math.log2(L)
    return {"bytes": 8 * n + 8 * Z * L + share * 4 * Z * n,
            "flops": nseg * 5 * L * lg + share * nseg * Z * (5 * L * lg + 6 * L + 3 * V)}


_LAYERS = 32 * 9 + 2 * 32 * 32 * 9   # multiply-adds per position of the three layers


def work(case):
    kind = case["kind"]
    if kind in ("plane", "fresh"):
        w = _plane_work(case["n"], 2 * (case["zmax"] // case["zstep"]) + 1, case["L"], case["m"])
        if kind == "fresh":   # the taps (a transform of the sampled chirp) and their spectra: made, not read
            w["flops"] += 2 * 5 * case["L"] * math.log2(case["L"]) * (2 * (case["zmax"] // case["zstep"]) + 1)
            w["bytes"] -= 8 * case["L"] * (2 * (case["zmax"] // case["zstep"]) + 1)
        return w
    if kind == "batch":
        n, zmax = _batch_sizes(case, 0)
        parts = [_plane_work(int(k), 2 * (int(z) // 2) + 1, case["L"], case["m"]) for k, z in zip(n, zmax)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "propose":
        nb = -(-case["n"] // zband.HOP)
        return {"bytes": 8 * case["n"] + 4 * nb * case["Z"],
                "flops": 2 * (_LAYERS * case["n"] + 32 * nb * case["Z"])}
    if kind == "pairs":
        Z = 2 * (case["zmax"] // case["zstep"]) + 1
        mask = _pair_mask(case, _logits(case, 1))
        w = _plane_work(case["n"], Z, 2048, 512, float(mask.float().mean()))
        w["bytes"] += 4 * Z * -(-case["n"] // zband.HOP) + 4 * int(mask.sum())
        return w
    B, Z, W = case["batch"], case["Z"], zband.WINDOW
    # forward; backward of weights and of data, whose pooled gradient is sparse before layer 3
    dense = 2 * 32 * 32 * 9 * W * B
    return {"bytes": 4 * B * (W + Z) + 4 * 8 * (_LAYERS + 33 * Z),
            "flops": 2 * (_LAYERS * W * B + dense + 32 * 9 * W * B + 3 * 32 * Z * B)}


# ----------------------------------------------------------------------------------------------
# the same outputs in 64 bits
# ----------------------------------------------------------------------------------------------
def _taps(zmax, zstep, m):
    """Normalised H_q(z) = int_0^1 exp(i pi (z u^2 - (z + 2 q) u)) du, q = -m/2..m/2, by composite
    Gauss-Legendre quadrature: [Z, m + 1] complex128."""
    xg, wg = np.polynomial.legendre.leggauss(16)
    panels = int(zmax + m) + 8
    u = torch.from_numpy(((np.arange(panels)[:, None] + 0.5 + 0.5 * xg[None]) / panels).ravel()).to(DEV)
    w = torch.from_numpy(np.tile(0.5 * wg / panels, panels)).to(DEV)
    z = torch.arange(-zmax, zmax + 1, zstep, device=DEV, dtype=torch.float64)
    q = torch.arange(-(m // 2), m // 2 + 1, device=DEV, dtype=torch.float64)
    chirp = torch.polar(w.expand(z.numel(), -1).contiguous(), math.pi * z[:, None] * (u * u - u)[None])
    wave = torch.polar(torch.ones((), device=DEV, dtype=torch.float64).expand(u.numel(), q.numel()).contiguous(),
                       -2 * math.pi * torch.remainder(u[:, None] * q[None], 1.0))
    H = chirp @ wave
    return H / H.abs().square().sum(1, keepdim=True).sqrt()


def _exact_plane(spec, zmax, zstep, m):
    """|sum_q A_{r+q} conj(Hn_q(z))|^2, one zero-padded circular correlation per template."""
    n, h = spec.shape[0], m // 2
    N = 1 << (n + 2 * h - 1).bit_length()
    A = torch.fft.fft(torch.view_as_complex(spec.double().contiguous()), N)
    taps = _taps(zmax, zstep, m)
    out = torch.empty((taps.shape[0], n), device=DEV, dtype=torch.float64)
    at = torch.arange(-h, h + 1, device=DEV) % N
    t = torch.zeros(N, device=DEV, dtype=torch.complex128)
    for i in range(taps.shape[0]):
        t[at] = taps[i]
        y = torch.fft.ifft(A * torch.fft.fft(t).conj())[:n]
        out[i] = y.real.square() + y.imag.square()
    return out


def _pair_mask(case, logits):
    """[segments, templates]: listed pairs of the proposal (see zband_work_pairs)."""
    V, h, H = 1536, 256, zband.HOP
    nseg, nb = -(-case["n"] // V), logits.shape[0]
    low = -math.inf
    own = torch.full((nseg, logits.shape[1]), low, device=DEV)
    reach = own.clone()
    s = torch.arange(nseg, device=DEV)
    lo, hi = s * V, (s + 1) * V
    for k in range(-1, V // H + 2):
        w = lo // H + k
        ok = (w >= 0) & (w < nb)
        v = logits[w.clamp(0, nb - 1)]
        is_own = ok & (w * H < hi) & ((w + 1) * H > lo)
        is_reach = ok & ~is_own & (w * H < hi + h) & ((w + 1) * H > lo - h)
        own = torch.where(is_own[:, None], torch.maximum(own, v), own)
        reach = torch.where(is_reach[:, None], torch.maximum(reach, v), reach)
    f = (own >= np.float32(math.log(THRESHOLD / (1 - THRESHOLD)))) | (reach >= np.float32(math.log(REACH / (1 - REACH))))
    return torch.nn.functional.max_pool1d(f.float()[:, None], 2 * HALO + 1, 1, HALO)[:, 0] > 0


def _split_params(p, Z):
    p = torch.from_numpy(p.astype(np.float64)).to(DEV)
    C, K = 32, 9
    out, at = [], 0
    for shape in ((C, 1, K), (C,), (C, C, K), (C,), (C, C, K), (C,), (Z, C), (Z,)):
        k = math.prod(shape)
        out.append(p[at:at + k].reshape(shape).clone())
        at += k
    return out


def _layers(x, P, pad):
    for k, d in enumerate((1, 4, 16)):
        x = torch.relu(torch.nn.functional.conv1d(x, P[2 * k], P[2 * k + 1], dilation=d, padding=4 * d if pad else 0))
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("plane", "fresh"):
        return _exact_plane(_spectrum(case["n"], case["zmax"], seed), case["zmax"], case["zstep"], case["m"])
    if kind == "batch":
        n, zmax = _batch_sizes(case, seed)
        return [_exact_plane(_spectrum(int(k), int(z), seed + 7 * i), int(z), 2, case["m"])
                for i, (k, z) in enumerate(zip(n, zmax))]
    if kind == "pairs":
        plane = _exact_plane(_spectrum(case["n"], case["zmax"], seed), case["zmax"], case["zstep"], 512)
        mask = _pair_mask(case, _logits(case, seed))
        for z in range(plane.shape[0]):   # cells of other pairs are never written
            plane[z] *= mask[:, z].double().repeat_interleave(1536)[:case["n"]]
        return {"pairs": None, "plane": plane}
    if kind == "propose":
        P = _split_params(_params(case["Z"], seed).astype(np.float16).astype(np.float32), case["Z"])
        H, nb = zband.HOP, -(-case["n"] // zband.HOP)
        x = torch.nn.functional.pad(_power_x(_spectrum(case["n"], 200, seed)), (84, 84 + nb * H - case["n"]))
        out = torch.empty((nb, case["Z"]), device=DEV, dtype=torch.float64)
        for b in range(0, nb, 512):   # bands of blocks, to bound the memory
            e = min(nb, b + 512)
            h3 = _layers(x[b * H:e * H + 168].reshape(1, 1, -1), P, False)[0]
            out[b:e] = h3.reshape(32, e - b, H).amax(2).T @ P[6].T + P[7]
        return out
    W = zband.WINDOW
    p0 = _params(case["Z"], seed)
    P = [t.requires_grad_() for t in _split_params(p0, case["Z"])]
    win, lab = _windows(case, seed)
    h3 = _layers(win.double()[:, None], P, True)
    logits = h3[:, :, W // 4:3 * W // 4].amax(2) @ P[6].T + P[7]
    loss = torch.nn.functional.binary_cross_entropy_with_logits(logits, lab.double())
    g = torch.cat([t.reshape(-1) for t in torch.autograd.grad(loss, P)])
    # first Adam step: both moments are their bias corrections times g and g^2
    p1 = torch.cat([t.detach().reshape(-1) for t in P]) - 1e-3 * g / (g.abs() + 1e-8)
    return {"loss": float(loss.detach()), "grads": g.cpu().numpy(), "params": p1.cpu().numpy()}
