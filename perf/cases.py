"""The performance cases of this framework: the calls its users make, from the
smallest to the largest, as data (`listed`, `draw`), inputs and handles
(`prepare`), one pass through the public entry points (`run`), the work that a
pass cannot do without (`work`) and its value in 64 bits (`exact`).

Kinds of case and what they stand for:

deepclean  gw_deepclean_forward on a batch of overlapping windows of one
           recording: offline cleaning, and the latency of one window.
stream     gw_stream_push of n snapshots into a stream in its steady state
           (ring update, DeepClean on every window, subtraction and
           aggregation), device buffers: online cleaning (few snapshots per
           push) and bulk re-processing (64 per push).
detect     gw_whiten and gw_bbhnet_score on a batch of two-detector segments:
           the detection stage, alone (one segment) and in bulk.
train      the differentiable path: gw_trainer_forward, gw_band_loss,
           gw_band_loss_backward, gw_trainer_backward; loss and gradients of
           one optimiser step.
fir        gw_whiten and gw_fir_backward on long series: whitening a
           recording, and its backward.
serve      gw_server_replay of a few snapshots of every stream of a serving
           loop (host buffers in and out, ring update to logit).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2108_12430_gb300 import gwstream as G
from paper_2108_12430_gb300 import synth

CHANNELS = 21   # witness channels per detector
FS = 4096.0     # detector rate; whitening and detection run at FS / 2
NFFT = 8192
SERVE_WARM_ROUNDS = 20  # snapshots of every stream before the measured pass: whitened strain has reached BBHnet

PRECISION = {"fp32": G.GW_FP32, "bf16": G.GW_BF16, "fp8": G.GW_FP8}


# ---- the cases ----------------------------------------------------------------

def listed():
    return [
        # one second of one detector, as soon as it is there
        dict(name="deepclean fp32 1x4096", kind="deepclean", precision="fp32", batch=1, length=4096, step=256),
        dict(name="deepclean bf16 1x4096", kind="deepclean", precision="bf16", batch=1, length=4096, step=256),
        # online cleaning: one new snapshot of an 8 s window
        dict(name="stream bf16 push 1", kind="stream", precision="bf16", snapshots=1, window=32768, stride=256,
             average=True, delay=32512),
        # bulk re-processing: 64 snapshots of 8 s windows, full overlap-add
        dict(name="stream fp32 push 64", kind="stream", precision="fp32", snapshots=64, window=32768, stride=256,
             average=True, delay=32512),
        dict(name="stream bf16 push 64", kind="stream", precision="bf16", snapshots=64, window=32768, stride=256,
             average=True, delay=32512),
        # detection on one second of two detectors, and in bulk
        dict(name="detect bf16 1", kind="detect", precision="bf16", batch=1, length=2048),
        dict(name="detect fp32 256", kind="detect", precision="fp32", batch=256, length=2048),
        dict(name="detect bf16 256", kind="detect", precision="bf16", batch=256, length=2048),
        dict(name="detect fp8 256", kind="detect", precision="fp8", batch=256, length=2048),
        # regular retraining: the gradient of one step, in FP32 and on the tensor cores
        dict(name="train fp32 32x8192", kind="train", precision="fp32", batch=32, length=8192, checkpoint=False),
        dict(name="train bf16 32x8192", kind="train", precision="bf16", batch=32, length=8192, checkpoint=False),
        # the serving loop: four snapshots of each of 64 streams of uneven strides
        dict(name="serve bf16 64 streams", kind="serve", precision="bf16", streams=64, rounds=4, window=32768,
             strides="128,256,512"),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["deepclean", "deepclean", "stream", "stream", "detect", "detect", "detect", "train", "train",
                       "fir", "serve"])
    if kind == "deepclean":
        return dict(kind=kind, precision=rng.choice(["fp32", "bf16"]), batch=_log(rng, 1, 64),
                    length=8 * _log(rng, 128, 4096), step=_log(rng, 64, 600))
    if kind == "stream":
        stride = rng.choice([128, 192, 256, 512])
        window = stride * max(4, _log(rng, 4096, 32768) // stride)
        average = rng.random() < 0.7
        return dict(kind=kind, precision=rng.choice(["fp32", "bf16"]), snapshots=_log(rng, 1, 64), window=window,
                    stride=stride, average=average,
                    delay=window - stride if rng.random() < 0.5 else rng.randint(0, window - stride))
    if kind == "detect":
        length = 16 * _log(rng, 32, 192)
        return dict(kind=kind, precision=rng.choice(["fp32", "bf16", "fp8"]),
                    batch=_log(rng, 1, min(256, 256 * 2048 // length)), length=length)
    if kind == "train":
        return dict(kind=kind, precision=rng.choice(["fp32", "bf16"]), batch=_log(rng, 1, 32),
                    length=8 * rng.randint(288, 1024), checkpoint=rng.random() < 0.3)
    if kind == "fir":
        return dict(kind=kind, rows=_log(rng, 1, 64), taps=rng.choice([127, 513, 1025, 2049]),
                    length=_log(rng, 4096, 32768))
    return dict(kind="serve", precision=rng.choice(["fp32", "bf16"]), streams=_log(rng, 1, 64), rounds=rng.randint(1, 4),
                window=rng.choice([8192, 16384, 32768]), strides=rng.choice(["128,256,512", "256", "512,128"]))


# ---- inputs -------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _noise(gen, shape, amplitude):
    """Gaussian noise with the given amplitude spectral shape (a function of
    frequency / sample rate), float64, periodic along its last axis."""
    n = shape[-1]
    white = torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64)
    return torch.fft.irfft(torch.fft.rfft(white) * amplitude(torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64)), n=n)


def _psd_amplitude(fs):
    def amplitude(f):
        psd = synth.aligo_psd((f * fs).cpu().numpy())
        return torch.from_numpy(np.sqrt(psd * fs / 2.0)).to(f.device)
    return amplitude


def _witness(gen, rows, n):
    """[rows][CHANNELS][n] FP32: low-passed noise of unit variance; three
    channels carry the 60 Hz line."""
    x = _noise(gen, (rows, CHANNELS, n), lambda f: (1.0 + (f * FS / 256.0) ** 8) ** -0.5)
    t = torch.arange(n, device="cuda", dtype=torch.float64) / FS
    phase = torch.rand(rows, 3, 1, generator=gen, device="cuda", dtype=torch.float64) * 2 * math.pi
    x[:, :3] = 0.3 * x[:, :3] / x[:, :3].std(-1, keepdim=True) + torch.sin(2 * math.pi * 60.0 * t + phase)
    x = x - x.mean(-1, keepdim=True)
    return (x / x.std(-1, keepdim=True)).float()


def _strain(gen, witness):
    """[rows][n] FP32 at FS: coloured noise plus the line coupled in from the
    first three witness channels."""
    rows, _, n = witness.shape
    gain = 0.5 + torch.rand(3, generator=gen, device="cuda", dtype=torch.float64)
    return (_noise(gen, (rows, n), _psd_amplitude(FS)) + 0.2 * (witness[:, :3].double() * gain[:, None]).sum(1)).float()


def _segments(gen, batch, n):
    """[batch][2][n] FP32 at FS / 2: coloured noise, and a chirp in both
    detectors of half of the segments."""
    fs = FS / 2
    x = _noise(gen, (batch, 2, n), _psd_amplitude(fs))
    t = torch.arange(n, device="cuda", dtype=torch.float64) / fs
    u = torch.rand(batch, 4, generator=gen, device="cuda", dtype=torch.float64)
    tc = (0.25 + 0.5 * u[:, :1]) * n / fs
    f = (30.0 * ((tc - t).clamp_min(1e-4) / 0.5) ** -0.375).clamp_max(300.0)
    chirp = torch.exp(-0.5 * ((t - tc) / (0.1 + 0.2 * u[:, 1:2])) ** 2) * torch.sin(2 * math.pi * torch.cumsum(f, -1) / fs)
    on = (torch.arange(batch, device="cuda") % 2 == 0).double()[:, None]
    amplitude = on * (0.2 + 0.3 * u[:, 2:3])
    return (x + torch.stack([chirp * amplitude, chirp * amplitude * (0.5 + 0.5 * u[:, 3:4])], 1)).float()


class State:
    """Handles and buffers of one case; the library's objects are destroyed
    with it, in the reverse order of their creation."""

    def __init__(self):
        self.objects = []
        self.context = self.keep(G.gw_ctx_create(torch.cuda.current_device(), 0), G.gw_ctx_destroy)

    def keep(self, handle, destroy):
        self.objects.append((destroy, handle))
        return handle

    def model(self, kind, precision, params, **more):
        n_in = CHANNELS if kind == G.GW_MODEL_DEEPCLEAN else 2
        return self.keep(G.gw_model_create(self.context, kind, PRECISION[precision], n_in, params, **more),
                         G.gw_model_destroy)

    def __del__(self):
        torch.cuda.synchronize()
        while self.objects:
            destroy, handle = self.objects.pop()
            destroy(handle)


def _cuda_stream():
    return torch.cuda.current_stream().cuda_stream


def _psd(fs):
    return synth.psd_grid(fs, NFFT)[1]


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def run(state):
    return state.run()


def work(case):
    return globals()["_work_" + case["kind"]](case)


def exact(case, seed):
    with torch.no_grad():
        return globals()["_exact_" + case["kind"]](case, seed)


# ---- the networks in 64 bits ----------------------------------------------------

def _weights(layers):
    return [{k: torch.from_numpy(np.asarray(v, np.float64)).cuda() for k, v in p.items()} for p in layers]


def _layer(x, p, spec):
    kind, _, _, _, stride, left, right, out_pad, bn, act = spec
    if kind == "conv":
        y = F.conv1d(F.pad(x, (left, right)), p["w"], p["b"], stride=stride)
    else:
        y = F.conv_transpose1d(x, p["w"], p["b"], stride=stride, padding=left, output_padding=out_pad)
    if bn:
        scale = p["gamma"] / torch.sqrt(p["var"] + 1e-5)
        y = (y - p["mean"][:, None]) * scale[:, None] + p["beta"][:, None]
    return torch.tanh(y) if act == "tanh" else torch.relu(y) if act == "relu" else y


def _deepclean64(x, params):
    for p, spec in zip(params, synth.DEEPCLEAN_LAYERS):
        x = _layer(x, p, spec)
    return x[:, 0]


def _deepclean64_batched(x, params, size):
    return torch.cat([_deepclean64(x[i:i + size].double(), params) for i in range(0, x.shape[0], size)])


def _bbhnet64(x, layers, head, seen=None):
    """Logits; `seen` receives the largest magnitude of every conv layer's
    input (of a block's output for its shortcut) and of the last output."""
    specs = synth.bbhnet_layers()
    seen = [] if seen is None else seen
    top = lambda v: float(v.abs().max())  # noqa: E731
    seen.append(top(x))
    h = _layer(x, layers[0], specs[0])
    for block in range(4):
        i = 1 + 3 * block
        a = _layer(h, layers[i], specs[i])
        shortcut = _layer(h, layers[i + 2], specs[i + 2])
        out = torch.relu(_layer(a, layers[i + 1], specs[i + 1]) + shortcut)
        seen += [top(h), top(a), max(top(shortcut), top(out))]
        h = out
    seen.append(top(h))
    return h.mean(-1) @ head["w"].reshape(-1) + head["b"]


def _hann(n):
    k = torch.arange(n, dtype=torch.float64, device="cuda")
    return 0.5 * (1.0 - torch.cos(2.0 * math.pi * k / (n - 1)))


def _zero_phase(amplitude, taps):
    """Centred, Hann-windowed truncation of the inverse DFT of real amplitudes."""
    h = torch.fft.irfft(torch.from_numpy(np.asarray(amplitude, np.float64)).cuda() + 0j, n=NFFT)
    c = (taps - 1) // 2
    return torch.roll(h, c)[:taps] * _hann(taps)


def _whitening(fs, taps):
    return _zero_phase(np.sqrt(2.0 / (fs * _psd(fs))), taps)


def _loss_filter(taps):
    f, psd = synth.psd_grid(FS, NFFT)
    ramp = np.clip(np.minimum(f - 55.0, 65.0 - f) / 2.0, 0.0, 1.0)
    band = 0.5 * (1.0 - np.cos(math.pi * ramp))
    return _zero_phase(np.sqrt(band * np.interp(60.0, f, psd) / psd), taps)


def _correlate(x, h):
    """Valid-mode y[n] = sum_k h[k] x[n + k] along the last axis."""
    n = x.shape[-1]
    y = torch.fft.irfft(torch.fft.rfft(x, n=n) * torch.fft.rfft(h, n=n).conj(), n=n)
    return y[..., :n - h.shape[0] + 1]


def _deepclean_flops(length):
    total, n = 0, length
    for kind, cin, cout, k, stride, *_ in synth.DEEPCLEAN_LAYERS:
        out = n // stride if kind == "conv" else n * stride
        total += 2 * cin * cout * k * (out if kind == "conv" else n)
        n = out
    return total


def _bbhnet_flops(length):
    total, n = 0, length
    specs = synth.bbhnet_layers()
    total += 2 * specs[0][1] * specs[0][2] * specs[0][3] * n
    for block in range(4):
        n //= 2
        for _, cin, cout, k, *_ in specs[1 + 3 * block:4 + 3 * block]:
            total += 2 * cin * cout * k * n
    return total


# ---- deepclean -------------------------------------------------------------------

def _deepclean_inputs(case, seed):
    n = case["length"] + (case["batch"] - 1) * case["step"]
    return _witness(_generator(seed), 1, n)[0].contiguous()


class _DeepClean(State):
    def __init__(self, case, seed):
        super().__init__()
        self.case = case
        self.x = _deepclean_inputs(case, seed)
        self.y = torch.empty(case["batch"], case["length"], device="cuda")
        self.net = self.model(G.GW_MODEL_DEEPCLEAN, case["precision"], synth.flatten_params(synth.deepclean_params(seed)))

    def run(self):
        c = self.case
        G.gw_deepclean_forward(self.net, self.x.data_ptr(), self.x.shape[1], c["step"], c["batch"], c["length"],
                               self.y.data_ptr(), _cuda_stream())
        return self.y


_prepare_deepclean = _DeepClean


def _work_deepclean(case):
    n = case["length"] + (case["batch"] - 1) * case["step"]
    return {"bytes": 4 * (CHANNELS * n + case["batch"] * case["length"]),
            "flops": case["batch"] * _deepclean_flops(case["length"])}


def _exact_deepclean(case, seed):
    x = _deepclean_inputs(case, seed)
    windows = x.unfold(1, case["length"], case["step"]).transpose(0, 1)
    return _deepclean64_batched(windows, _weights(synth.deepclean_params(seed)), 16)


# ---- stream ----------------------------------------------------------------------

def _stream_pushes(case):
    """Pushes before the measured one: until the ring holds a whole window."""
    return -(-case["window"] // (case["snapshots"] * case["stride"]))


def _stream_inputs(case, seed):
    gen = _generator(seed)
    n = case["snapshots"] * case["stride"]
    witness = _witness(gen, 1, (_stream_pushes(case) + 1) * n)
    return witness[0], _strain(gen, witness)[0]


class _Stream(State):
    def __init__(self, case, seed):
        super().__init__()
        self.case = case
        net = self.model(G.GW_MODEL_DEEPCLEAN, case["precision"], synth.flatten_params(synth.deepclean_params(seed)))
        self.stream = self.keep(
            G.gw_stream_create(self.context, [net], 1, CHANNELS, case["window"], case["stride"], case["snapshots"],
                               G.GW_AGG_AVERAGE if case["average"] else G.GW_AGG_LATEST, case["delay"]),
            G.gw_stream_destroy)
        witness, strain = _stream_inputs(case, seed)
        n = case["snapshots"] * case["stride"]
        self.clean = torch.empty(1, n, device="cuda")
        for k in range(_stream_pushes(case) + 1):
            self.witness = witness[:, k * n:(k + 1) * n].contiguous()
            self.strain = strain[k * n:(k + 1) * n].contiguous()
            if k < _stream_pushes(case):
                self.run()
        torch.cuda.synchronize()

    def run(self):
        G.gw_stream_push(self.stream, self.case["snapshots"], self.witness.data_ptr(), self.strain.data_ptr(),
                         self.clean.data_ptr(), G.GW_MEM_DEVICE, _cuda_stream())
        return self.clean


_prepare_stream = _Stream


def _work_stream(case):
    n, s, w = case["snapshots"], case["stride"], case["window"]
    size = 4 if case["precision"] == "fp32" else 2
    # new samples in, the windows' ring read once, predictions aggregated into the stream's state, cleaned samples out
    return {"bytes": 4 * (CHANNELS + 2) * n * s + size * CHANNELS * (w + (n - 1) * s) + 8 * (w + n * s),
            "flops": n * _deepclean_flops(w)}


def _exact_stream(case, seed):
    w, s, n, delay = case["window"], case["stride"], case["snapshots"], case["delay"]
    witness, strain = _stream_inputs(case, seed)
    before = _stream_pushes(case) * n
    total = before + n
    first, end = before * s - delay, total * s - delay  # the times that the measured push emits
    padded = F.pad(witness, (w - s, 0))                 # zeros before the stream
    params = _weights(synth.deepclean_params(seed))
    prediction = torch.zeros(end - first, dtype=torch.float64, device="cuda")
    if case["average"]:
        # window k covers the times [(k + 1) s - w, (k + 1) s); a time counts the windows pushed when it is emitted
        count = torch.zeros_like(prediction)
        at = torch.arange(first, end, device="cuda")
        emitted_at = (at + delay) // s
        ks = list(range(max(0, first // s), total))
        for i in range(0, len(ks), 16):
            some = ks[i:i + 16]
            out = _deepclean64(torch.stack([padded[:, k * s:k * s + w] for k in some]).double(), params)
            for k, p in zip(some, out):
                offset = at - ((k + 1) * s - w)
                on = (offset >= 0) & (offset < w) & (emitted_at >= k)
                prediction += torch.where(on, p[offset.clamp(0, w - 1)], 0.0)
                count += on
        prediction /= count
    else:
        for i in range(before, total, 16):
            some = range(i, min(i + 16, total))
            out = _deepclean64(torch.stack([padded[:, k * s:k * s + w] for k in some]).double(), params)
            for k, p in zip(some, out):
                prediction[(k - before) * s:(k - before + 1) * s] = p[w - s - delay:w - delay]
    clean = torch.where(torch.arange(first, end, device="cuda") >= 0,
                        strain.double()[torch.arange(first, end, device="cuda").clamp_min(0)], 0.0)
    return (clean - prediction)[None]


# ---- detect ----------------------------------------------------------------------

DETECT_TAPS = 2049


def _fp8_scales(layers, head, length):
    """Static activation scales, as a user gets them from a calibration batch."""
    x = _segments(_generator(7), 16, length + DETECT_TAPS - 1).double()
    seen = []
    _bbhnet64(_correlate(x, _whitening(FS / 2, DETECT_TAPS)), _weights(layers), _weights([head])[0], seen)
    return np.array([448.0 / (1.25 * v) for v in seen], np.float32)


class _Detect(State):
    def __init__(self, case, seed):
        super().__init__()
        self.case = case
        b, n = case["batch"], case["length"]
        self.x = _segments(_generator(seed), b, n + DETECT_TAPS - 1)
        self.white = torch.empty(b, 2, n, device="cuda")
        self.logits = torch.empty(b, device="cuda")
        layers, head = synth.bbhnet_params(seed)
        scales = _fp8_scales(layers, head, n) if case["precision"] == "fp8" else None
        self.net = self.model(G.GW_MODEL_BBHNET, case["precision"], synth.flatten_params(layers, head), act_scales=scales)
        self.fir = self.keep(
            G.gw_fir_create_whitening(self.context, _psd(FS / 2), FS / 2, DETECT_TAPS,
                                      G.GW_FP32 if case["precision"] == "fp32" else G.GW_BF16), G.gw_fir_destroy)

    def run(self):
        b, n, stream = self.case["batch"], self.case["length"], _cuda_stream()
        G.gw_whiten(self.fir, self.x.data_ptr(), b, 2, n + DETECT_TAPS - 1, self.white.data_ptr(), stream)
        G.gw_bbhnet_score(self.net, self.white.data_ptr(), b, n, self.logits.data_ptr(), stream)
        return {"whitened": self.white, "logits": self.logits}


_prepare_detect = _Detect


def _work_detect(case):
    b, n = case["batch"], case["length"]
    return {"bytes": 4 * b * (2 * (n + DETECT_TAPS - 1) + 2 * n + 1),
            "flops": b * (_bbhnet_flops(n) + 2 * 2 * DETECT_TAPS * n)}


def _exact_detect(case, seed):
    x = _segments(_generator(seed), case["batch"], case["length"] + DETECT_TAPS - 1)
    white = _correlate(x.double(), _whitening(FS / 2, DETECT_TAPS))
    layers, head = synth.bbhnet_params(seed)
    layers, head = _weights(layers), _weights([head])[0]
    return {"whitened": white, "logits": torch.cat([_bbhnet64(v, layers, head) for v in white.split(32)])}


# ---- train -----------------------------------------------------------------------

TRAIN_TAPS = 2049


def _train_inputs(case, seed):
    gen = _generator(seed)
    x = _witness(gen, case["batch"], case["length"])
    return x.contiguous(), _strain(gen, x).contiguous()


class _Train(State):
    def __init__(self, case, seed):
        super().__init__()
        self.case = case
        b, n = case["batch"], case["length"]
        self.x, self.strain = _train_inputs(case, seed)
        self.params = torch.from_numpy(synth.flatten_params(synth.deepclean_params(seed))).cuda()
        tensor_cores = case["precision"] == "bf16"
        self.trainer = self.keep(
            G.gw_trainer_create(self.context, CHANNELS, b, n, int(case["checkpoint"]),
                                precision=PRECISION[case["precision"]], tc_data=int(tensor_cores)), G.gw_trainer_destroy)
        self.fir = self.keep(G.gw_fir_create_band_loss(self.context, _psd(FS), FS, TRAIN_TAPS), G.gw_fir_destroy)
        self.y, self.dy = torch.empty(b, n, device="cuda"), torch.empty(b, n, device="cuda")
        self.residual = torch.empty(b, n - TRAIN_TAPS + 1, device="cuda")
        self.loss = torch.empty(1, device="cuda")
        self.gradient = torch.empty_like(self.params)

    def run(self):
        b, n, stream = self.case["batch"], self.case["length"], _cuda_stream()
        G.gw_trainer_forward(self.trainer, self.params.data_ptr(), self.x.data_ptr(), b, self.y.data_ptr(), stream)
        G.gw_band_loss(self.fir, self.strain.data_ptr(), self.y.data_ptr(), b, n, self.loss.data_ptr(),
                       self.residual.data_ptr(), stream)
        G.gw_band_loss_backward(self.fir, self.residual.data_ptr(), b, n, 0, self.dy.data_ptr(), stream)
        G.gw_trainer_backward(self.trainer, self.dy.data_ptr(), self.gradient.data_ptr(), stream)
        return {"prediction": self.y, "loss": self.loss, "gradient": self.gradient}


_prepare_train = _Train


def _work_train(case):
    b, n = case["batch"], case["length"]
    first = 2 * CHANNELS * 8 * 7 * n  # the network's input needs no gradient
    return {"bytes": 4 * b * n * (CHANNELS + 2) + 3 * 4 * 39041,
            "flops": b * (3 * _deepclean_flops(n) - first + 2 * 2 * TRAIN_TAPS * (n - TRAIN_TAPS + 1))}


def _exact_train(case, seed):
    x, strain = _train_inputs(case, seed)
    raw = synth.deepclean_params(seed)
    params = _weights(raw)
    names = [(i, k) for i, p in enumerate(raw) for k in synth.PARAM_ORDER if k in p]
    trained = [(i, k) for i, k in names if k not in ("mean", "var")]
    for i, k in trained:
        params[i][k].requires_grad_()
    with torch.enable_grad():
        y = _deepclean64(x.double(), params)
        loss = _correlate(strain.double() - y, _loss_filter(TRAIN_TAPS)).square().mean()
        gradients = dict(zip(trained, torch.autograd.grad(loss, [params[i][k] for i, k in trained])))
    flat = torch.cat([gradients.get((i, k), torch.zeros_like(params[i][k])).reshape(-1) for i, k in names])
    return {"prediction": y.detach(), "loss": loss.detach().reshape(1), "gradient": flat}


# ---- fir -------------------------------------------------------------------------

def _fir_inputs(case, seed):
    gen = _generator(seed)
    n = case["length"]
    x = _noise(gen, (case["rows"], n), _psd_amplitude(FS / 2)).float().contiguous()
    return x, torch.randn(case["rows"], n - case["taps"] + 1, generator=gen, device="cuda")


class _Fir(State):
    def __init__(self, case, seed):
        super().__init__()
        self.case = case
        self.x, self.dy = _fir_inputs(case, seed)
        self.y, self.dx = torch.empty_like(self.dy), torch.empty_like(self.x)
        self.fir = self.keep(G.gw_fir_create_whitening(self.context, _psd(FS / 2), FS / 2, case["taps"]), G.gw_fir_destroy)

    def run(self):
        rows, n, stream = self.case["rows"], self.case["length"], _cuda_stream()
        G.gw_whiten(self.fir, self.x.data_ptr(), rows, 1, n, self.y.data_ptr(), stream)
        G.gw_fir_backward(self.fir, self.dy.data_ptr(), rows, 1, n, self.dx.data_ptr(), stream)
        return {"whitened": self.y, "dx": self.dx}


_prepare_fir = _Fir


def _work_fir(case):
    rows, n, k = case["rows"], case["length"], case["taps"]
    return {"bytes": 4 * rows * (4 * n - 2 * (k - 1)), "flops": 2 * 2 * rows * k * (n - k + 1)}


def _exact_fir(case, seed):
    x, dy = _fir_inputs(case, seed)
    k = case["taps"]
    h = _whitening(FS / 2, k)
    return {"whitened": _correlate(x.double(), h), "dx": _correlate(F.pad(dy.double(), (k - 1, k - 1)), h.flip(0))}


# ---- serve -----------------------------------------------------------------------

SERVE_SCORE = 2048  # BBHnet's input length
DECIMATOR_TAPS, WHITENING_TAPS = 127, 2049


def _serve_strides(case):
    strides = [int(s) for s in case["strides"].split(",")]
    return [strides[i % len(strides)] for i in range(case["streams"])]


def _serve_inputs(case, seed):
    """Per stride: its streams, and witness [round][stream][2][C][S] and strain
    [round][stream][2][S] of a series that repeats after `rounds` snapshots."""
    gen = _generator(seed)
    rounds, per_stream, got = case["rounds"], _serve_strides(case), {}
    for s in sorted(set(per_stream)):
        ids = [i for i, v in enumerate(per_stream) if v == s]
        w = _witness(gen, 2 * len(ids), rounds * s)
        x = _strain(gen, w)
        w = w.reshape(len(ids), 2, CHANNELS, rounds, s).permute(3, 0, 1, 2, 4)
        x = x.reshape(len(ids), 2, rounds, s).permute(2, 0, 1, 3)
        got[s] = (ids, w, x)
    return got


def _serve_params(seed):
    """Both detectors' DeepClean (its output layer scaled to the strain, as
    training would) and BBHnet."""
    cleaners = []
    for d in range(2):
        p = synth.deepclean_params(seed + d)
        p[-1] = {k: (v * np.float32(1e-2)).astype(np.float32) for k, v in p[-1].items()}
        cleaners.append(p)
    return cleaners, synth.bbhnet_params(seed + 2)


class _Serve(State):
    def __init__(self, case, seed):
        super().__init__()
        cleaners, (layers, head) = _serve_params(seed)
        nets = [self.model(G.GW_MODEL_DEEPCLEAN, case["precision"], synth.flatten_params(p)) for p in cleaners]
        bbh = self.model(G.GW_MODEL_BBHNET, case["precision"], synth.flatten_params(layers, head))
        dec = self.keep(G.gw_fir_create_lowpass(self.context, 900.0, FS, DECIMATOR_TAPS), G.gw_fir_destroy)
        white = self.keep(G.gw_fir_create_whitening(self.context, _psd(FS / 2), FS / 2, WHITENING_TAPS), G.gw_fir_destroy)
        n, rounds = case["streams"], case["rounds"]
        per_stream = _serve_strides(case)
        self.server = self.keep(
            G.gw_server_create(self.context, nets, bbh, dec, white, n_det=2, n_witness=CHANNELS, window=case["window"],
                               max_stride=max(per_stream), max_streams=n, max_batch=n, max_pending=4 * n,
                               agg_mode=G.GW_AGG_AVERAGE, agg_delay=0, bbh_len=SERVE_SCORE), G.gw_server_destroy)
        opened = [G.gw_server_open(self.server, s) for s in per_stream]
        self.inputs, self.clean = [], {}
        addresses = np.zeros((3, rounds, n), np.uint64)
        for s, (ids, w, x) in _serve_inputs(case, seed).items():
            w, x = w.contiguous().cpu().numpy(), x.contiguous().cpu().numpy()
            self.clean[s] = np.zeros_like(x)
            self.inputs += [w, x]
            for j, a in enumerate((w, x, self.clean[s])):
                at = a.ctypes.data + a[0, 0].nbytes * np.arange(rounds * len(ids), dtype=np.uint64)
                addresses[j][:, ids] = at.reshape(rounds, len(ids))
        self.addresses = addresses.reshape(3, -1).copy()
        self.ids = np.tile(np.array(opened, np.int32), rounds)
        self.due = np.zeros(rounds * n)  # every snapshot is there: the loop's throughput
        self.scores = np.zeros(rounds * n, np.float32)
        for _ in range(-(-SERVE_WARM_ROUNDS // rounds)):
            self.run()

    def run(self):
        G.gw_server_replay(self.server, self.ids, self.due, *self.addresses, self.scores)
        return {"clean": {str(s): v for s, v in self.clean.items()}, "logits": self.scores}


_prepare_serve = _Serve


def _work_serve(case):
    n = sum(_serve_strides(case)) * case["rounds"]
    count = case["streams"] * case["rounds"]
    size = 4 if case["precision"] == "fp32" else 2
    return {"bytes": 2 * 4 * n * (CHANNELS + 2) + count * (2 * case["window"] * (size * CHANNELS + 8) + 8 * SERVE_SCORE),
            "flops": count * (2 * _deepclean_flops(case["window"]) + _bbhnet_flops(SERVE_SCORE))}


def _exact_serve(case, seed):
    cleaners, (layers, head) = _serve_params(seed)
    layers, head = _weights(layers), _weights([head])[0]
    cleaners = [_weights(p) for p in cleaners]
    rounds, n = case["rounds"], case["streams"]
    cycles = 1 + -(-SERVE_WARM_ROUNDS // rounds)  # passes through the series, the measured one last
    total = cycles * rounds
    margin = 512  # more samples than an output sees to its left
    c = (DECIMATOR_TAPS - 1) / 2.0
    k = torch.arange(DECIMATOR_TAPS, dtype=torch.float64, device="cuda") - c
    low = 2 * 900.0 / FS * torch.sinc(2 * 900.0 / FS * k) * _hann(DECIMATOR_TAPS)
    low = low / low.sum()
    white = _whitening(FS / 2, WHITENING_TAPS)
    clean_out, logits = {}, torch.zeros(rounds, n, dtype=torch.float64, device="cuda")
    for s, (ids, w, x) in _serve_inputs(case, seed).items():
        w = w.permute(1, 2, 3, 0, 4).reshape(len(ids), 2, CHANNELS, rounds * s).repeat(1, 1, 1, cycles)
        x = x.permute(1, 2, 0, 3).reshape(len(ids), 2, rounds * s).repeat(1, 1, cycles).double()
        padded = F.pad(w, (margin, 0))
        predicted = torch.zeros_like(x)
        for d in range(2):
            crops = padded[:, d].unfold(2, margin + s, s).permute(0, 2, 1, 3).reshape(-1, CHANNELS, margin + s)
            predicted[:, d] = _deepclean64_batched(crops, cleaners[d], 256)[:, margin:].reshape(len(ids), total * s)
        clean = x - predicted
        clean_out[str(s)] = clean.reshape(len(ids), 2, total, s)[:, :, -rounds:].permute(2, 0, 1, 3)
        half = (DECIMATOR_TAPS - 1) // 2
        low_rate = _correlate(F.pad(clean, (half, half)), low)[..., ::2]
        for r in range(rounds):
            known = (total - rounds + r + 1) * s
            m_end = (known - 64) // 2 + 1 if known >= 64 else 0
            n_end = m_end - (WHITENING_TAPS - 1) // 2
            score = torch.zeros(len(ids), 2, SERVE_SCORE, dtype=torch.float64, device="cuda")
            if n_end > 0:
                w_all = _correlate(F.pad(low_rate[..., :m_end], ((WHITENING_TAPS - 1) // 2, 0)), white)[..., :n_end]
                some = min(n_end, SERVE_SCORE)
                score[..., SERVE_SCORE - some:] = w_all[..., n_end - some:]
            logits[r, torch.tensor(ids, device="cuda")] = _bbhnet64(score, layers, head)
    return {"clean": clean_out, "logits": logits.reshape(-1)}
