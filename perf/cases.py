"""The calls whose speed this repository measures, with their inputs and their values in 64 bits.

Every case goes through the package's public classes as a user's program calls them, with the handles, models and
output buffers that such a program keeps. The sizes are those of the bench, the tests and the paper's defaults (batches
of 128 voices of 4 s at 44.1 kHz; inverse synthesis on 64 voices of 1 s; corpora of 1024 sounds each); draw() spreads
over the same ranges, odd and ragged sizes among them.

The 64-bit values are plain torch in float64 on the GPU: the Voice and the FM voice by their definitions, the adjoint by
autograd, the spectra by torch.stft."""
import math

import numpy as np
import torch

import paper_2104_12922_gb300 as pkg

CONTROL_RATE = 441
STEPS = 4  # training steps between two looks at the weights


def listed():
    return [
        # one sound on demand, as an instrument or a listening page asks for it: the smallest call
        {"name": "voice_1", "kind": "render", "batch": 1, "samples": 176400, "rate": 44100},
        # one replicable batch of the paper's default size, one call for each batch
        {"name": "batch_128", "kind": "render", "batch": 128, "samples": 176400, "rate": 44100},
        # corpus generation at full speed: consecutive batches in one launch, as the bench times it
        {"name": "batches_20x128", "kind": "batches", "batch": 128, "count": 20, "samples": 176400, "rate": 44100},
        # a corpus without silent or quiet sounds: peak normalisation and rejection
        {"name": "normalized_128", "kind": "normalized", "batch": 128, "samples": 176400, "rate": 44100},
        # speech-rate corpora: a fractional number of samples per control interval
        {"name": "rate16k_128", "kind": "render", "batch": 128, "samples": 64000, "rate": 16000},
        # the second architecture, the 4-operator FM voice
        {"name": "fm_128", "kind": "fm", "batch": 128, "samples": 176400, "rate": 44100},
        # inverse synthesis by gradient descent: the render's adjoint
        {"name": "adjoint_64", "kind": "adjoint", "batch": 64, "samples": 44100, "rate": 44100},
        # ... and its loss with the gradient, against targets seen before
        {"name": "mrstft_64", "kind": "mrstft", "batch": 64, "samples": 44100, "rate": 44100, "target_ready": True},
        # network input features of a rendered batch
        {"name": "logmel_128", "kind": "logmel", "batch": 128, "samples": 176400, "rate": 44100},
        # parameters proposed for a handful of recorded sounds
        {"name": "propose_16", "kind": "propose", "batch": 16, "samples": 176400, "rate": 44100},
        # training of the proposal network on features in hand
        {"name": "train_128", "kind": "train", "batch": 128, "samples": 176400, "rate": 44100},
        # similarity of three corpora: pairwise distances of their features (the largest)
        {"name": "distances_3072", "kind": "distances", "batch": 3072, "dim": 44160},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "batches", "normalized", "fm", "adjoint", "mrstft", "logmel", "propose",
                       "train", "distances"])
    if kind == "distances":
        return {"kind": kind, "batch": _log(rng, 48, 3000), "dim": 128 * _log(rng, 22, 345)}
    rate = rng.choice([44100, 44100, 16000, 22050, 48000]) if kind in ("render", "normalized", "fm") else 44100
    case = {"kind": kind, "batch": _log(rng, 1, 128), "samples": _log(rng, rate // 4, 4 * rate), "rate": rate}
    if kind == "batches":
        case.update(batch=_log(rng, 16, 128), count=rng.randint(2, 19))
    elif kind == "adjoint":
        case.update(batch=_log(rng, 1, 64), samples=_log(rng, 4410, 88200))
    elif kind == "mrstft":
        case.update(batch=_log(rng, 1, 64), samples=_log(rng, 4410, 88200), target_ready=rng.random() < 0.5)
    elif kind in ("propose", "train"):
        case["batch"] = 8 * _log(rng, 1, 16)
    return case


# ---- what a program has in hand ---------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _sounds(batch, samples, rate, seed):
    """Sounds [batch][samples] like the Voice's: decaying gliding partials and noise from near silence to full scale,
    a part of them ending in digital silence. Elementwise in the sample index."""
    g = _gen(seed)

    def u(lo, hi):
        return lo + (hi - lo) * torch.rand(batch, 1, generator=g, device="cuda", dtype=torch.float64)

    t = torch.arange(samples, device="cuda", dtype=torch.float64) / rate
    f0, glide = 27.5 * 2 ** u(0, 8), u(-0.3, 0.3)
    phase = f0 * t * (1 + 0.5 * glide * t)
    x = torch.zeros(batch, samples, device="cuda", dtype=torch.float64)
    for k in range(1, 7):
        fades = torch.where(f0 * k * 1.6 < rate / 2, torch.exp(-t * u(0, 6)), 0.0)
        x += u(0, 1) / k * fades * torch.sin(2 * math.pi * (k * phase + u(0, 1)))
    noise = torch.randn(batch, samples, generator=g, device="cuda", dtype=torch.float64)
    x += u(0.05, 0.5) ** 2 * noise * torch.exp(-t * u(0, 4))
    x *= 10 ** u(-3, 0) / 2
    return torch.where(t < u(0.3, 2.0) * samples / rate, x, 0.0).float()


def _embeddings(m, dim, seed):
    """Log-mel embeddings [m][dim] (bands minor) of m sounds in the features' range: a spectrum for each sound with its
    decay, the roughness of single frames, a floor, and some silent sounds (all at the floor)."""
    g = _gen(seed)

    def u(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda")

    frames = dim // 128
    floor = (math.log(1e-6) - pkg.FEATURE_SHIFT) / pkg.FEATURE_SCALE
    out = torch.empty(m, dim, device="cuda", dtype=torch.bfloat16)
    for at in range(0, m, 256):
        n = min(256, m - at)
        band = torch.arange(128, device="cuda") / 127
        tone = torch.exp(-((band - u(0, 1, n, 1)) / u(0.02, 0.6, n, 1)) ** 2)
        level = u(-1.5, 1.6, n, 1, 1) + u(0, 1.5, n, 1, 1) * tone[:, None, :]
        fade = u(0, 3, n, 1, 1) * torch.linspace(0, 1, frames, device="cuda")[None, :, None]
        e = level - fade + 0.2 * torch.randn(n, frames, 128, generator=g, device="cuda")
        e = torch.clamp(e, min=floor)
        e[torch.rand(n, generator=g, device="cuda") < 0.03] = floor
        out[at:at + n] = e.reshape(n, dim).bfloat16()
    return out


def _uniform(batch, count, seed):
    """Normalized parameters, 24-bit as the library draws them."""
    return torch.randint(0, 1 << 24, (batch, count), generator=_gen(seed), device="cuda").float() / (1 << 24)


def _training_set(case, seed):
    """STEPS batches of features of sounds with the parameters to learn."""
    frames = 1 + case["samples"] // 512
    feats = _embeddings(STEPS * case["batch"], 128 * frames, seed).view(STEPS, case["batch"], -1)
    return feats, _uniform(STEPS * case["batch"], pkg.NUM_PARAMS, seed + 1).view(STEPS, case["batch"], -1)


def _first_batch(seed):
    return 1000 + seed % 100000


def prepare(case, seed):
    kind, batch = case["kind"], case["batch"]
    s = {"case": case, "seed": seed}
    if kind == "distances":
        s["synth"] = pkg.Synth(max_batch=1)
        s["emb"] = _embeddings(batch, case["dim"], seed)
        s["out"] = torch.empty(batch, batch, device="cuda")
        return s
    total = batch * case.get("count", 1)
    s["synth"] = pkg.Synth(seconds=case["samples"] / case["rate"], sample_rate=float(case["rate"]),
                           control_rate=float(CONTROL_RATE), max_batch=8 * ((total + 7) // 8))
    if kind in ("render", "batches", "normalized", "fm"):
        s["out"] = torch.empty(total, case["samples"], device="cuda")
        s["params"] = torch.empty(total, pkg.FM_NUM_PARAMS if kind == "fm" else pkg.NUM_PARAMS, device="cuda")
    elif kind == "adjoint":
        s["params"] = _uniform(batch, pkg.NUM_PARAMS, seed)
        s["grad_audio"] = torch.randn(batch, case["samples"], generator=_gen(seed + 1), device="cuda")
    elif kind == "mrstft":
        s["x"] = _sounds(batch, case["samples"], case["rate"], seed)
        s["y"] = _sounds(batch, case["samples"], case["rate"], seed + 1)
        s["mr"] = pkg.MRSTFT(s["synth"], batch)
        if case["target_ready"]:
            s["mr"](s["x"], s["y"], grad=False)
    else:
        s["model"] = pkg.ProposalModel(s["synth"], max_batch=8 * ((batch + 7) // 8), seed=seed)
        if kind == "train":
            s["feats"], s["target"] = _training_set(case, seed)
            s["loss"] = torch.empty(STEPS, device="cuda")
        else:
            s["audio"] = _sounds(batch, case["samples"], case["rate"], seed)
    return s


def run(s):
    case, seed, syn = s["case"], s["seed"], s["synth"]
    kind, batch = case["kind"], case["batch"]
    if kind == "render":
        audio, params = syn.render(seed, _first_batch(seed), batch, out=s["out"], params_out=s["params"])
        return {"audio": audio, "params": params}
    if kind == "batches":
        audio, params = syn.render_batches(seed, 1, _first_batch(seed), batch, case["count"], out=s["out"],
                                           params_out=s["params"])
        return {"audio": audio, "params": params}
    if kind == "normalized":
        audio, params, peak, silent = syn.render_normalized(seed, _first_batch(seed), batch, out=s["out"],
                                                            params_out=s["params"])
        return {"audio": audio, "params": params, "peak": peak, "silent": silent}
    if kind == "fm":
        audio, params = syn.fm_render(seed, _first_batch(seed), batch, out=s["out"], params_out=s["params"])
        return {"audio": audio, "params": params}
    if kind == "adjoint":
        return {"grad": syn.backward(seed, _first_batch(seed), s["params"], s["grad_audio"])}
    if kind == "mrstft":
        loss, grad = s["mr"](s["x"], s["y"], target_ready=case["target_ready"])
        return {"loss": loss, "grad": grad}
    if kind == "logmel":
        return {"features": s["model"].features(s["audio"])}
    if kind == "propose":
        return {"params": s["model"].propose(s["audio"])}
    if kind == "train":
        for i in range(STEPS):
            s["model"].train_features(s["feats"][i], s["target"][i], 1e-4, loss=s["loss"][i:i + 1])
        out = {"loss": s["loss"]}
        for layer in range(4):
            out["w%d" % layer] = s["model"].tensor(0, layer)
            out["b%d" % layer] = s["model"].tensor(1, layer)
        return out
    return {"dist": pkg.l1_distances(syn, s["emb"], out=s["out"])}


# ---- what a pass cannot do without ------------------------------------------------------------------------------------
def work(case):
    kind, batch = case["kind"], case["batch"]
    if kind == "distances":
        # a subtraction and an addition for each pair of elements of two different sounds
        return {"bytes": 2 * batch * case["dim"] + 4 * batch * batch, "flops": batch * (batch - 1) * case["dim"]}
    n = case["samples"]
    frames = 1 + n // 512
    points = batch * case.get("count", 1) * n
    if kind in ("render", "batches", "normalized", "fm"):
        # audio written once (and, normalized, scaled in place); about 60 operations for each sample
        return {"bytes": (12 if kind == "normalized" else 4) * points, "flops": 60 * points}
    if kind == "adjoint":
        return {"bytes": 4 * points + 8 * 78 * batch, "flops": 120 * points}
    if kind == "mrstft":
        # three resolutions at a hop of a quarter: four transforms' worth of points each way
        each = sum(4 * 2.5 * math.log2(w) for w in (512, 1024, 2048))
        return {"bytes": (12 + (0 if case["target_ready"] else 4)) * points,
                "flops": (2 if case["target_ready"] else 3) * each * points}
    dims = [128 * frames, 1024, 1024, 1024, 78]
    weights = sum(a * b for a, b in zip(dims, dims[1:]))
    fft = batch * frames * 2.5 * 2048 * 11
    if kind == "logmel":
        return {"bytes": 4 * points + 256 * batch * frames, "flops": fft}
    if kind == "propose":
        return {"bytes": 4 * points + 2 * weights, "flops": fft + 2 * batch * weights}
    # a training step reads the bf16 weights, and reads and writes the weights, both moments and the copy
    return {"bytes": STEPS * (2 * weights + 26 * weights + 2 * batch * dims[0]) + 8 * weights,
            "flops": STEPS * (6 * batch * weights - 2 * batch * dims[0] * dims[1])}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    low = 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2  # wraps mod 2^64: all 64 bits are the product's
        c0, c1, c2, c3 = ((p1 >> 32) & low) ^ c1 ^ k0, p1 & low, ((p0 >> 32) & low) ^ c3 ^ k1, p0 & low
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c0, c1, c2, c3


def _draws(seeds, g, count, stream):
    """`count` uniform values for each voice g [B] under its seed: [B][count], multiples of 2^-24."""
    block = torch.arange((count + 3) // 4, device=g.device)[None, :]
    gg, ss = g[:, None], seeds[:, None]
    words = _philox(gg & 0xFFFFFFFF, gg >> 32, block, torch.full_like(block, stream), ss & 0xFFFFFFFF, ss >> 32)
    words = [w.expand(g.shape[0], block.shape[1]) for w in words]
    return (torch.stack(words, 2).reshape(g.shape[0], -1)[:, :count] >> 8).double() / (1 << 24)


def _ranges():
    adsr = [(0, 2, 2), (0, 2, 2), (0, 1, 1), (0, 5, 2), (0.1, 6, 2)]
    pi = math.pi
    r = [(0, 127, 1, 0), (0, 4, 1, 0)] + [x + (0,) for x in 6 * adsr]
    r += 2 * ([(0, 20, 2, 0), (-20, 20, 3, 1), (-pi, pi, 1, 1)] + 5 * [(0, 1, 1, 0)]) + 20 * [(0, 1, 2, 0)]
    r += 2 * [(-24, 24, 1, 1), (-96, 96, 3, 1), (-pi, pi, 1, 1)] + [(0, 1, 1, 0)] + 3 * [(0, 1, 1, 0)]
    return r


def _fm_ranges():
    adsr = [(0, 2, 2), (0, 2, 2), (0, 1, 1), (0, 5, 2), (0.1, 6, 2)]
    r = [(0, 127, 1), (0, 4, 1)]
    for i in range(4):
        r += [(0.5, 8, 2), (0, 1, 1) if i == 0 else (0, 8, 2)] + adsr
    return [x + (0,) for x in r]


def _pow(x, a):
    pos = x > 0
    return torch.where(pos, torch.where(pos, x, 1.0) ** a, 0.0)


def _map(u, ranges):
    lo, hi, c, sym = (torch.tensor(v, dtype=torch.float64, device=u.device) for v in zip(*ranges))
    s = 2 * u - 1
    bent = (1 + torch.sign(s) * _pow(s.abs(), c)) / 2
    return lo + (hi - lo) * torch.where(sym > 0, bent, _pow(u, c))


def _over(x, y):
    return x / torch.where(y > 0, y, 1.0)


def _adsr(t, q, d):
    a, dc, s, r, alpha = (q[:, i:i + 1] for i in range(5))

    def gate(x):
        return torch.where(x < a, _pow(_over(x, a), alpha),
                           torch.where(x < a + dc, 1 - (1 - s) * _pow(_over(x - a, dc), alpha), s))

    after = torch.where(t - d < r, gate(d) * (1 - _pow(_over(t - d, r), alpha)), 0.0)
    return torch.where(t < d, gate(t), after)


def _frac(x):
    return x - torch.floor(x)


def _running(x):
    """Sums of all earlier values."""
    return torch.cumsum(x, 1) - x


def _grid(samples, rate, device):
    """Each sample's control interval and its place in it, and the times of the control points."""
    n = torch.arange(samples, device=device)
    k = n * CONTROL_RATE // rate
    t = torch.arange(int(k[-1]) + 2, device=device, dtype=torch.float64) / CONTROL_RATE
    return k, (n * CONTROL_RATE - k * rate).double() / rate, t[None, :]


def _voice(u, seeds, g, samples, rate):
    """Audio of voices with normalized parameters u [B][78]: [B][samples]."""
    y = _map(u, _ranges())
    k, at, t = _grid(samples, rate, u.device)
    col = lambda i: y[:, i:i + 1]  # noqa: E731
    env = [_adsr(t, y[:, 2 + 5 * a:7 + 5 * a], col(1)) for a in range(6)]
    lfo = []
    for i in range(2):
        b = 32 + 8 * i
        hz = torch.clamp(col(b) + col(b + 1) * env[2 + 2 * i], 0.0, 20.0)
        p = _frac(col(b + 2) / (2 * math.pi) + _running(hz / CONTROL_RATE))
        shapes = [torch.sin(2 * math.pi * p), 1 - 4 * (p - 0.5).abs(), 2 * p - 1, 1 - 2 * p,
                  torch.where(p < 0.5, 1.0, -1.0).to(p)]
        total = y[:, b + 3:b + 8].sum(1, keepdim=True)
        mixed = sum(col(b + 3 + j) * shapes[j] for j in range(5)) / torch.clamp(total, min=1e-12)
        lfo.append(env[3 + 2 * i] * torch.where(total >= 1e-12, mixed, 0.0))
    src = [env[0], env[1], lfo[0], lfo[1]]

    def dest(j):
        w = [col(48 + 5 * i + j) for i in range(4)]
        return sum(a * b for a, b in zip(w, src)) / torch.clamp(sum(w), min=1.0)

    def up(c):
        c0 = c[:, k]
        return c0 + at * (c[:, k + 1] - c0)

    nyquist = 69 + 12 * math.log2(rate / 2 / 440)

    def hz(m):
        return 440 * torch.exp2((torch.clamp(m, max=nyquist) - 69) / 12)

    def phase(m, b):
        return 2 * math.pi * _frac(col(b + 2) / (2 * math.pi) + _running(hz(up(m)) / rate))

    level = [col(75), col(76), col(77)]
    norm = torch.clamp(sum(level), min=1.0)
    out = level[0] / norm * up(dest(1)) * torch.sin(phase(col(0) + col(68) + col(69) * dest(0), 68))
    m = col(0) + col(71) + col(72) * dest(2)
    theta = phase(m, 71)
    kappa = torch.clamp(1 + rate / 8 / hz(m), max=50.0)[:, k]
    square = torch.tanh(kappa * torch.sin(theta)) / torch.tanh(kappa)
    out = out + level[1] / norm * up(dest(3)) * square * (1 + col(74) * torch.cos(theta)) / (1 + col(74))
    noise = 2 * _draws(seeds, g, samples, 1) - 1
    return out + level[2] / norm * up(dest(4)) * noise


def _fm_voice(u, samples, rate):
    y = _map(u, _fm_ranges())
    k, at, t = _grid(samples, rate, u.device)
    n = torch.arange(samples, device=u.device, dtype=torch.float64)
    f0 = 440 * torch.exp2((y[:, 0:1] - 69) / 12)
    out = 0.0
    for i in (3, 2, 1, 0):
        q = y[:, 2 + 7 * i:9 + 7 * i]
        env = _adsr(t, q[:, 2:7], y[:, 1:2])
        e = env[:, k] + at * (env[:, k + 1] - env[:, k])
        out = q[:, 1:2] * e * torch.sin(2 * math.pi * _frac(n * (f0 * q[:, 0:1] / rate)) + out)
    return out


def _stft(x, size, hop):
    w = torch.hann_window(size, periodic=True, dtype=torch.float64, device=x.device)
    return torch.stft(x, size, hop_length=hop, window=w, center=True, pad_mode="reflect", return_complex=True)


def _distance(x, y):
    total = 0.0
    for size in (512, 1024, 2048):
        a, b = (torch.log(_stft(v, size, size // 4).abs() + 1e-7) for v in (x, y))
        total = total + (a - b).abs().mean(dim=(1, 2))
    return total


def _mel_bank(rate):
    """Triangles of unit area, their edges equally spaced on the Slaney mel scale: [128][1025]."""
    top = 15 + 27 * math.log(rate / 2 / 1000) / math.log(6.4)
    mel = np.linspace(0, top, 130)
    edge = np.where(mel < 15, 200 * mel / 3, 1000 * np.exp((mel - 15) * math.log(6.4) / 27))
    bins = np.arange(1025) * rate / 2048
    lo, mid, hi = (edge[i:i + 128, None] for i in range(3))
    bank = np.maximum(0, np.minimum((bins - lo) / (mid - lo), (hi - bins) / (hi - mid))) * 2 / (hi - lo)
    return torch.from_numpy(bank).cuda()


def _features(audio, rate):
    bank, out = _mel_bank(rate), []
    for part in audio.split(16):
        power = _stft(part.double(), 2048, 512).abs() ** 2
        mel = torch.matmul(bank, power).transpose(1, 2)
        out.append(((torch.log(mel + 1e-6) - pkg.FEATURE_SHIFT) / pkg.FEATURE_SCALE).flatten(1))
    return torch.cat(out)


def _network(frames, seed):
    """The weights and biases that a new model of this seed starts with."""
    dims = [128 * frames, 1024, 1024, 1024, 78]
    key = torch.tensor(seed, device="cuda")
    w = []
    for layer in range(4):
        block = torch.arange(dims[layer] * dims[layer + 1] // 4, device="cuda")
        none = torch.zeros_like(block)
        words = torch.stack(_philox(block, none + layer, none, none + 2, key & 0xFFFFFFFF, key >> 32), 1)
        bound = torch.tensor(1.0 / math.sqrt(dims[layer]), dtype=torch.float32).item()
        v = bound * (2 * (words >> 8).double() / (1 << 24) - 1)
        w.append(v.float().double().reshape(dims[layer + 1], dims[layer]))
    return w, [torch.zeros(n, device="cuda", dtype=torch.float64) for n in dims[1:]]


def _forward(x, w, b):
    for layer in range(4):
        x = x @ w[layer].T + b[layer]
        x = torch.sigmoid(x) if layer == 3 else torch.relu(x)
    return x


def _train(case, seed):
    frames = 1 + case["samples"] // 512
    w, b = _network(frames, seed)
    feats, target = _training_set(case, seed)
    every = [v.requires_grad_(True) for v in w + b]
    m, v = [torch.zeros_like(p) for p in every], [torch.zeros_like(p) for p in every]
    losses = []
    for step in range(STEPS):
        loss = ((_forward(feats[step].double(), w, b) - target[step].double()) ** 2).mean()
        losses.append(loss.detach())
        for i, g in enumerate(torch.autograd.grad(loss, every)):
            m[i].mul_(0.9).add_(0.1 * g)
            v[i].mul_(0.999).add_(0.001 * g * g)
            with torch.no_grad():
                every[i] -= 1e-4 * (m[i] / (1 - 0.9 ** (step + 1))) / (
                    torch.sqrt(v[i] / (1 - 0.999 ** (step + 1))) + 1e-8)
    out = {"loss": torch.stack(losses)}
    for layer in range(4):
        # Adam's first steps move a bias from its 0 by its gradient's sign alone, and the sign of a small sum turns on
        # the 16-bit activations
        out["w%d" % layer], out["b%d" % layer] = w[layer].detach(), None
    return out


def _rendered(case, seed):
    """Parameters and audio of the case's voices, some voices at a time."""
    batch, total, n = case["batch"], case["batch"] * case.get("count", 1), case["samples"]
    g = _first_batch(seed) * batch + torch.arange(total, device="cuda")
    seeds = seed + torch.arange(total, device="cuda") // batch
    fm = case["kind"] == "fm"
    u = _draws(seeds, g, 30 if fm else 78, 2 if fm else 0)
    audio = torch.empty(total, n, device="cuda", dtype=torch.float64)
    for at in range(0, total, 64):
        part = slice(at, min(total, at + 64))
        audio[part] = (_fm_voice(u[part], n, case["rate"]) if fm
                       else _voice(u[part], seeds[part], g[part], n, case["rate"]))
    return u, audio


def exact(case, seed):
    kind, batch = case["kind"], case["batch"]
    if kind == "distances":
        e = _embeddings(batch, case["dim"], seed).double()
        return {"dist": torch.stack([(e - e[i]).abs_().sum(1) for i in range(batch)])}
    if kind in ("render", "batches", "fm"):
        u, audio = _rendered(case, seed)
        return {"audio": audio, "params": u}
    if kind == "normalized":
        u, audio = _rendered(case, seed)
        peak = audio.abs().amax(1)
        loud = (peak >= 1e-3) & (peak > 0)
        scale = torch.where(loud, 1 / torch.where(loud, peak, 1.0), 1.0)
        return {"audio": audio * scale[:, None], "params": u, "peak": peak, "silent": None}
    if kind == "adjoint":
        grads = []
        u = _uniform(batch, pkg.NUM_PARAMS, seed).double()
        w = torch.randn(batch, case["samples"], generator=_gen(seed + 1), device="cuda").double()
        g = _first_batch(seed) * batch + torch.arange(batch, device="cuda")
        seeds = torch.full_like(g, seed)
        for at in range(0, batch, 32):
            part = slice(at, min(batch, at + 32))
            v = u[part].clone().requires_grad_(True)
            audio = _voice(v, seeds[part], g[part], case["samples"], case["rate"])
            grads.append(torch.autograd.grad((audio * w[part]).sum(), v)[0])
        return {"grad": torch.cat(grads)}
    if kind == "mrstft":
        x = _sounds(batch, case["samples"], case["rate"], seed).double()
        y = _sounds(batch, case["samples"], case["rate"], seed + 1).double()
        loss, grad = [], []
        for a, b in zip(x.split(16), y.split(16)):
            a = a.clone().requires_grad_(True)
            each = _distance(a, b)
            loss.append(each.detach())
            grad.append(torch.autograd.grad(each.sum(), a)[0])
        return {"loss": torch.cat(loss), "grad": torch.cat(grad)}
    if kind == "train":
        return _train(case, seed)
    feats = _features(_sounds(batch, case["samples"], case["rate"], seed), case["rate"])
    if kind == "logmel":
        return {"features": feats}
    w, b = _network(1 + case["samples"] // 512, seed)
    return {"params": _forward(feats, w, b)}
