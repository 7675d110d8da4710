"""Performance cases of the mixing-console library: the calls that its users make, through the public Python API
(paper_2509_15948_gb300.Console), from the smallest console to a batch of songs.

A case names what is run ("kind"), the console (songs, tracks, subgroups, lengths, sample rate, processor types,
loss settings) and the option in use.  Inputs come from the seed: synthetic multitrack audio (pink-noise bursts and
decaying notes), a target mix of the same tracks with other gains, a spectral tilt and a reverberant tail, and
processor parameters over the ranges that a search visits.

  step    one training step as the search runs it (Sec. 5.1): forward, loss, backward and Adam, replayed as one
          CUDA graph; set_params first, so that every pass trains from the same point
  crop    the same step on a new crop of the song (update_audio, then the step): the paper's training regime
  grad    the differentiable console as torch code uses it: set_params, forward_loss with the mixes, backward,
          get_grads
  render  a masked forward with the mixes, and the evaluation metrics of those mixes
  score   one call of batched pruning trials (Alg. 3): L_a of every song under every candidate mask
"""
import math
import random

import numpy as np
import torch

import paper_2509_15948_gb300 as M

ORDER = "ecnsgdr"
COUNT = {"e": 1024, "c": 4, "n": 4, "s": 1, "g": 2, "d": 880, "r": 768}
FS = 44100
ALPHA_P = 1e-4


# ---------------------------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------------------------

def _case(kind, types=ORDER, **kw):
    c = {"kind": kind, "types": types, "fs": FS, "fft0": 512, "fft1": 2048, "fft2": 8192, "songs": 1, "tracks": 1,
         "tracks_max": 0, "groups": 0, "samples": FS, "samples_max": 0, "layout": 0, "warmup": 0, "retain": 0,
         "graph": False, "nodes": 0, "masks": 0}
    c.update(kw)
    if not c["tracks_max"]:
        c["tracks_max"] = c["tracks"]
    if not c["samples_max"]:
        c["samples_max"] = c["samples"]
    return c


def listed():
    return [
        # the smallest console that the tests and the benchmark run (4 tracks x 2 s, one subgroup): a step is
        # about a hundred short launches, so latency and launch counts decide
        _case("step", name="plain_step", tracks=4, groups=1, samples=2 * FS),
        # one song of the single-song search (16 tracks x 10 s in 4 subgroups), the unit of a search
        _case("step", name="song_step", tracks=16, groups=4, samples=10 * FS),
        # songs of uneven sizes trained together, as the batched search and the benchmark's default do
        _case("step", name="batch_step", songs=10, tracks=4, tracks_max=32, groups=8, samples=5 * FS,
              samples_max=30 * FS, layout=2),
        # the paper's training regime: 3.8 s crops at 30 kHz, its STFT sizes, the first second left out of the loss
        _case("crop", name="crop_step", fs=30000, fft1=1024, fft2=4096, tracks=24, groups=4, samples=114000,
              warmup=30000),
        # a long song under the serving loop's setting, the FFT spectra recomputed in the backward
        _case("grad", name="long_recompute", tracks=8, groups=2, samples=60 * FS - 77, retain=-1),
        # one processor type at a time: reverbs (a 2 s FIR per track) ...
        _case("grad", "r", name="reverb_block", tracks=12, groups=0, samples=12 * FS + 1003),
        # ... multitap delays ...
        _case("grad", "d", name="delay_block", tracks=12, groups=3, samples=7 * FS + 211),
        # ... equalizers (2047 taps) with the panning that a stereo mix has ...
        _case("grad", "eg", name="equalizer_block", tracks=24, groups=4, samples=10 * FS + 37),
        # ... compressors and gates (a scan along the whole signal), a short odd length and few tracks ...
        _case("grad", "cng", name="dynamics_block", tracks=6, groups=0, samples=5 * FS + 129),
        # ... and gain, panning and imaging with the loss, which is most of a lightly processed song
        _case("grad", "gs", name="balance_block", tracks=24, groups=6, samples=30 * FS + 5),
        # pruning trials of one search round
        _case("score", name="prune_trials", tracks=16, groups=4, samples=10 * FS, masks=16),
        # rendering a pruned song and measuring it
        _case("render", name="render_metrics", tracks=20, groups=4, samples=19 * FS + 401),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "batch", "crop", "long", "block", "block", "block", "graph", "score", "render"])
    if kind == "step":
        k = rng.randint(1, 24)
        return _case("step", tracks=k, groups=rng.randint(0, min(k, 6)), samples=_log(rng, FS // 2, 20 * FS))
    if kind == "batch":
        return _case("step", songs=rng.randint(2, 8), tracks=rng.randint(1, 6), tracks_max=rng.randint(8, 24),
                     groups=rng.randint(1, 8), samples=_log(rng, FS, 6 * FS), samples_max=_log(rng, 8 * FS, 24 * FS),
                     layout=rng.randint(3, 1000))
    if kind == "crop":
        k = rng.randint(8, 32)
        return _case("crop", fs=30000, fft1=1024, fft2=4096, tracks=k, groups=rng.randint(1, 6),
                     samples=_log(rng, 75000, 180000), warmup=30000)
    if kind == "long":
        k = rng.randint(2, 8)
        return _case("grad", tracks=k, groups=rng.randint(0, 2), samples=_log(rng, 20 * FS, 60 * FS), retain=-1)
    if kind == "block":
        types = rng.choice(["r", "d", "eg", "cng", "gs", "cg", "er"])
        k = rng.randint(1, 24)
        return _case("grad", types, tracks=k, groups=rng.randint(0, min(k, 4)), samples=_log(rng, FS // 2, 25 * FS))
    if kind == "graph":
        # a general processing graph (Sec. 4) instead of the console
        return _case("grad", graph=True, tracks=rng.randint(2, 6), nodes=rng.randint(12, 30),
                     samples=_log(rng, FS, 12 * FS), layout=rng.randint(0, 1000))
    if kind == "score":
        k = rng.randint(2, 16)
        return _case("score", tracks=k, groups=rng.randint(0, min(k, 4)), samples=_log(rng, 2 * FS, 10 * FS),
                     masks=rng.randint(1, 20))
    k = rng.randint(1, 24)
    return _case("render", tracks=k, groups=rng.randint(0, min(k, 6)), samples=_log(rng, FS, 25 * FS))


def _songs(case):
    """[(tracks, subgroups, group of every track, samples)] of a case."""
    if case["songs"] == 1:
        k, s = case["tracks"], case["groups"]
        # a console with subgroups leaves its last track ungrouped when there are enough of them
        return [(k, s, [(-1 if (k > 2 * s and t == k - 1) else t % s) if s else -1 for t in range(k)], case["samples"])]
    r = random.Random(case["layout"])
    out = []
    for _ in range(case["songs"]):
        k = r.randint(case["tracks"], case["tracks_max"])
        s = min(k, r.randint(1, case["groups"]))
        out.append((k, s, [t % s for t in range(k)], r.randint(case["samples"], case["samples_max"])))
    return out


def _graph_of(case):
    """A general graph (node types, input tracks, edges): inputs, then processors of every type and two mix nodes in a
    shuffled order, each fed by one or two earlier nodes, and an output fed by every node that nothing reads."""
    r = random.Random(case["layout"])
    types, track, edges = [M.NODE_INPUT] * case["tracks"], list(range(case["tracks"])), []
    kinds = list(range(7)) + [r.randrange(7) for _ in range(case["nodes"] - 7)] + [M.NODE_MIX] * 2
    r.shuffle(kinds)
    for t in kinds:
        v = len(types)
        edges += [(u, v) for u in sorted({r.randrange(v) for _ in range(r.randint(1, 2))})]
        types.append(t)
        track.append(-1)
    read = {u for u, _ in edges}
    o = len(types)
    edges += [(v, o) for v in range(o) if v not in read]
    return types + [M.NODE_OUTPUT], track + [-1], edges


def _proc_types(case):
    """[(type, song)] of every processor in canonical order."""
    if case["graph"]:
        return [(ORDER[t], 0) for t in _graph_of(case)[0] if t < 7]
    return [(t, i) for i, (k, s, _, _) in enumerate(_songs(case)) for _ in range(k + s) for t in ORDER
            if t in case["types"]]


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------

def _gen(seed, *key):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + sum((k + 1) * 7919 ** i for i, k in enumerate(key))) & 0x7FFFFFFFFFFF)
    return g


def _tracks(g, k, n, fs):
    """[k][n] dry mono tracks on the GPU: pink-noise bursts plus decaying notes over a recording's noise floor, peak
    -6 dBFS."""
    def u(lo, hi, *shape):
        return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo
    spec = torch.fft.rfft(torch.randn(k, n, generator=g, device="cuda"))
    f = torch.arange(spec.shape[1], device="cuda", dtype=torch.float32).clamp(min=1.0)
    f[0] = float("inf")
    pink = torch.fft.irfft(spec / f.sqrt(), n=n)
    pink = pink / pink.std(dim=1, keepdim=True).clamp(min=1e-12)
    # on / off durations with mean 0.5 s, 5 ms ramps
    m = int(n / fs * 4) + 24
    ends = torch.cumsum(-0.5 * fs * torch.log(u(1e-6, 1.0, k, m)), 1)
    at = torch.arange(n, device="cuda", dtype=torch.float32).expand(k, n).contiguous()
    on = ((torch.searchsorted(ends, at) + (torch.arange(k, device="cuda") % 2)[:, None]) % 2).float()
    ramp = 2 * int(0.0025 * fs) + 1
    x = pink * torch.nn.functional.avg_pool1d(on[:, None], ramp, 1, ramp // 2, count_include_pad=False)[:, 0]
    x *= u(0.2, 1.0, k, 1)
    x += pink * 0.002
    notes = max(1, int(2 * n / fs))
    lvl = u(0.2, 1.0, k, 1)
    for _ in range(notes):
        t = (at - u(0.0, float(n), k, 1).floor()) / fs
        fr, tau, amp = torch.exp(u(4.0073, 7.4731, k, 1)), u(0.1, 1.0, k, 1), u(0.3, 1.0, k, 1)
        x += lvl * amp * torch.where(t >= 0, torch.sin(2 * math.pi * fr * t) * torch.exp(-t.clamp(min=0) / tau), 0.0)
    return (x * (0.501 / x.abs().amax(dim=1, keepdim=True).clamp(min=1e-9))).contiguous()


def _target(g, src, fs):
    """[2][n] finished mix of the tracks: other gains and pans, a spectral tilt, a reverberant tail."""
    k, n = src.shape
    gains = torch.exp(torch.rand(2, k, generator=g, device="cuda") * 1.5 - 1.0)
    m = 2 * n
    dry = torch.fft.rfft(gains @ src, n=m)
    f = torch.arange(dry.shape[1], device="cuda") * (fs / m)
    tilt = (1.0 + f / 2000.0) ** -0.4
    tail = torch.randn(2, n, generator=g, device="cuda") * torch.exp(-torch.arange(n, device="cuda") / (0.3 * fs)) * 0.02
    y = torch.fft.irfft(dry * tilt * (1.0 + torch.fft.rfft(tail, n=m)), n=m)[:, :n]
    return y.float().contiguous()


def _params(r, types):
    """Parameters of a search under way: every type over the range that it visits, logits of the dry/wet weights."""
    out = []
    for t in types:
        if t == "g":
            p = r.uniform(-1.0, 1.0, 2)
        elif t == "s":
            p = r.uniform(-1.0, 0.5, 1)
        elif t == "e":
            p = np.interp(np.arange(1024), np.linspace(0, 1023, 8), r.uniform(-1.0, 1.0, 8))
        elif t == "r":
            p = np.stack([r.uniform(-6.0, -3.0, (2, 192)), r.uniform(-1.0, 1.0, (2, 192))], 1).ravel()
        elif t in "cn":
            lo, hi = (-8.0, -2.0) if t == "c" else (-14.0, -8.0)
            p = np.array([r.uniform(4.0, 9.0), r.uniform(lo, hi), r.uniform(-1.0, 1.0), r.uniform(0.0, 2.0)])
        else:
            rad, ang = r.uniform(0.9, 1.0, (2, 20)), r.uniform(-np.pi, np.pi, (2, 20))
            p = np.concatenate([np.stack([rad * np.cos(ang), rad * np.sin(ang)], 2), r.uniform(-5.0, -3.0, (2, 20, 20))], 2).ravel()
        out.append(p)
    out.append(r.normal(0.0, 0.5, len(types)))
    return np.concatenate(out).astype(np.float32)


def _inputs(case, seed):
    fs, songs, types = case["fs"], _songs(case), [t for t, _ in _proc_types(case)]
    src, tgt = [], []
    for i, (k, _, _, n) in enumerate(songs):
        g = _gen(seed, i)
        full = n + (fs * 6 if case["kind"] == "crop" else 0)   # crops are cut from a longer song
        x = _tracks(g, k, full, fs)
        src.append(x)
        tgt.append(_target(g, x, fs))
    r = np.random.default_rng([seed & 0x7FFFFFFF, 17])
    nrev = sum(t == "r" for t in types)
    noise = torch.rand(nrev, 2, 2 * fs, generator=_gen(seed, 9001), device="cuda") * 2.0 - 1.0 if nrev else None
    params = _params(r, types)
    masks = None
    if case["kind"] == "score":    # a window of trials: each drops the least-weight few of one type
        masks = np.ones((case["masks"], len(types)), np.uint8)
        q = params[-len(types):]
        for j in range(case["masks"]):
            pick = types[r.integers(len(types))]
            same = sorted((i for i, t in enumerate(types) if t == pick), key=lambda i: q[i])
            masks[j, same[: int(r.integers(1, 4))]] = 0
    elif case["kind"] == "render":  # a pruned graph: about a third of the processors is left
        masks = (r.random(len(types)) < 0.4).astype(np.uint8)
    crop = int(r.integers(0, fs * 6 + 1)) if case["kind"] == "crop" else 0
    return src, tgt, noise, params, masks, crop


def prepare(case, seed):
    src, tgt, noise, params, masks, crop = _inputs(case, seed)
    songs = [M.Song(k, s, g, n) for k, s, g, n in _songs(case)]
    cfg = M.ConsoleConfig(sample_rate=float(case["fs"]), types=case["types"], n_fft=(case["fft0"], case["fft1"], case["fft2"]),
                          warmup_samples=case["warmup"], retain_spectra=case["retain"])
    graph = M.Graph(*_graph_of(case)) if case["graph"] else None
    n = [s.num_samples for s in songs]
    con = M.Console(songs, [x[:, :m] for x, m in zip(src, n)], [x[:, :m] for x, m in zip(tgt, n)], noise, cfg, graph=graph)
    con.set_alpha_p(ALPHA_P)
    p = torch.as_tensor(params, device="cuda")
    con.set_params(p)
    st = {"kind": case["kind"], "con": con, "params": p}
    if masks is not None:
        st["mask"] = torch.as_tensor(masks, device="cuda")
    if case["kind"] == "crop":
        st["crop"] = (src[0][:, crop:crop + n[0]], tgt[0][:, crop:crop + n[0]])
    torch.cuda.synchronize()
    return st


def run(state):
    con, kind = state["con"], state["kind"]
    if kind == "score":
        return {"la": con.prune_scores(state["mask"])}
    if kind == "render":
        losses, mixes = con.forward_loss(state["mask"], with_mix=True)
        return {"losses": losses, "mix": mixes, "metrics": con.evaluate()}
    con.set_params(state["params"])
    if kind == "grad":
        losses, mixes = con.forward_loss(with_mix=True)
        con.backward()
        return {"losses": losses, "mix": mixes, "grads": con.get_grads()}
    if kind == "crop":
        con.update_audio(0, *state["crop"])
    losses = con.train_step()
    return {"losses": losses.clone(), "grads": con.get_grads()}


# ---------------------------------------------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------

def work(case):
    """Five stereo FP32 streams per processor (the forward reads u and writes y, the backward reads dL/dy and u and
    writes dL/du; two without a backward), the sums and the loss on top; 2.5 n log2 n operations per real FFT of
    size n of the convolutions and of the STFTs, and twenty per sample of the other processors."""
    back = case["kind"] in ("step", "crop", "grad")
    times = max(1, case["masks"]) if case["kind"] == "score" else 1
    songs, stream, total, flops = _songs(case), 0.0, 0.0, 0.0
    per_song = [0] * len(songs)
    for t, i in _proc_types(case):
        n = songs[i][3]
        per_song[i] += 1
        total += (5 if back else 2) * 8.0 * n
        if t in "erd":
            m = 2047 + n if t == "e" else 2 * case["fs"] + n
            if t == "e":
                m, blocks = 8192, math.ceil(n / 6146)
            else:
                blocks = 1
            flops += blocks * 2 * 2.5 * m * math.log2(m) * (6 if back else 3)
        else:
            flops += 20.0 * 2 * n * (2 if back else 1)
    for k, s, _, n in songs:
        total += 8.0 * n * (1.5 * k + 2 * s + 4)
        for f in (case["fft0"], case["fft1"], case["fft2"]):
            flops += max(0, (n - f) // (f // 4) + 1) * 2 * 2.5 * f * math.log2(f) * (2 if back else 1)
    if case["kind"] == "score":    # a trial renders again only what its mask changes: a few chains and the mix
        k, s, _, n = songs[0]
        stream = 8.0 * n * (2 * 2 * len(set(case["types"])) + k + s + 4)
        share = 4.0 / max(1, k + s)
        return {"bytes": total + times * stream, "flops": flops * (1 + times * share)}
    return {"bytes": total, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------------------------------------------

D64 = torch.float64


def _conv(x, h, n0):
    """y[n] = sum_j h[j] x[n - n0 - j], n in [0, L), zero outside."""
    n = x.shape[-1]
    m = 1 << (n + h.shape[-1] - 1).bit_length()
    y = torch.fft.irfft(torch.fft.rfft(x, m) * torch.fft.rfft(h, m), m)
    return y[..., -n0:-n0 + n]


def _zero_phase(p, taps):
    """Zero-phase FIR of the log-magnitudes p (half of a mirrored response), windowed; first tap at -(taps - 1) / 2."""
    half = (taps - 1) // 2
    h = torch.fft.ifft(torch.exp(torch.cat([p, p[..., 1:].flip(-1)], -1)).to(torch.complex128)).real
    t = torch.arange(-half, half + 1, dtype=D64, device=p.device)
    return torch.roll(h, half, -1) * (0.5 + 0.5 * torch.cos(2 * math.pi * t / (taps - 1)))


def _hann(n):
    return 0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(n, dtype=D64, device="cuda") / n)


class _Taps(torch.autograd.Function):
    """The delay's FIR (one 39-tap FIR per tap, at integer delays) and the straight-through direction of its delays."""

    @staticmethod
    def forward(ctx, c, z, slot, n):
        ph = torch.remainder(-torch.atan2(z[..., 1], z[..., 0]), 2 * math.pi)
        at = torch.remainder(torch.round(slot * ph / (2 * math.pi)).long(), slot) + slot * torch.arange(20, device=z.device)
        h = torch.zeros(2, 20 * slot + 38, dtype=D64, device=z.device)
        idx = at[..., None] + torch.arange(39, device=z.device)
        for ch in range(2):
            h[ch].index_add_(0, idx[ch].reshape(-1), c[ch].reshape(-1))
        ctx.save_for_backward(c, z, idx)
        ctx.slot, ctx.n = slot, n
        return h

    @staticmethod
    def backward(ctx, dh):
        c, z, idx = ctx.saved_tensors
        slot = ctx.slot
        dc = torch.stack([dh[ch][idx[ch]] for ch in range(2)])
        dt = dh.clone()
        dt[:, ctx.n + 19:] = 0.0
        zc = torch.complex(z[..., 0], z[..., 1])
        r = zc.abs()
        zk = zc / r.clamp(min=1.0)
        k = torch.arange(slot, device=z.device, dtype=D64)
        a = torch.zeros(2, 20, slot, dtype=torch.complex128, device=z.device)
        a[..., 1:] = k[1:] * torch.exp((k[1:] - 1) * torch.log(zk)[..., None])
        ds = torch.fft.ifft(a)
        win = dt.unfold(1, 39, 1)[:, :20 * slot].reshape(2, 20, slot, 39)
        corr = torch.einsum("cmqj,cmj->cmq", win, c)
        g = (corr * ds.conj()).sum(-1)
        d = torch.where(g.abs() > 0, g / g.abs().clamp(min=1e-300), 0.0) + 0.01 * (r - 1.0) * zc / r.clamp(min=1e-300)
        return dc, torch.stack([d.real, d.imag], -1), None, None


def _reverb_taps(p, noise, length):
    win = _hann(384)
    u = torch.fft.rfft(noise.to(D64).unfold(-1, 384, 192) * win)         # [2][frames][193]
    f = u.shape[1]
    p = p.reshape(2, 2, 192)
    p = torch.cat([p, p[..., -1:]], -1)
    t = torch.arange(f, dtype=D64, device="cuda")[:, None]
    mask = torch.exp(p[:, 0, None] - 0.05 * t * torch.nn.functional.softplus(p[:, 1, None]))
    fr = torch.fft.irfft(u * mask, 384) * win
    n = 192 * (f + 1)

    def ola(x):
        y = torch.zeros(x.shape[0], n, dtype=D64, device="cuda")
        y = y + torch.nn.functional.pad(x[:, :, :192].reshape(x.shape[0], -1), (0, 192))
        return y + torch.nn.functional.pad(x[:, :, 192:].reshape(x.shape[0], -1), (192, 0))
    env = ola((win * win).expand(1, f, 384))
    h = ola(fr) / torch.where(env > 1e-11, env, torch.full_like(env, float("inf")))
    h = torch.nn.functional.pad(h, (0, length - n))
    return torch.stack([h[0] + h[1], h[0] - h[1]])


def _envelope_gain(u, p, gate):
    alpha, t, w, ratio = torch.sigmoid(p[0]), p[1], torch.exp(p[2]), 1 + torch.exp(p[3])
    k = torch.arange(u.shape[-1], dtype=D64, device="cuda")
    g = _conv((u[0] + u[1]) ** 2, torch.sigmoid(-p[0]) * torch.exp(k * torch.log(alpha)), 0)
    x = torch.log(g + 1e-8)
    if gate:
        y = torch.where(x >= t + w, x, torch.where(x >= t - w, x + (1 - ratio) * (x - t - w) ** 2 / (4 * w), t + ratio * (x - t)))
    else:
        y = torch.where(x >= t + w, t + (x - t) / ratio, torch.where(x >= t - w, x + (1 / ratio - 1) * (x - t + w) ** 2 / (4 * w), x))
    return torch.exp(y - x) * u


def _process(t, u, p, w, noise, fs):
    """(output of a processor with its dry/wet blend, its gain-staging term)."""
    lg = torch.zeros((), dtype=D64, device="cuda")
    if t == "g":
        y = torch.exp(p)[:, None] * u
    elif t == "s":
        m, s = u[0] + u[1], torch.exp(p[0]) * (u[0] - u[1])
        y = torch.stack([m + s, m - s]) / 2
    elif t in "cn":
        y = _envelope_gain(u, p, t == "n")
    else:
        if t == "e":
            y = _conv(u, _zero_phase(p, 2047)[None], -1023)
        elif t == "r":
            y = _conv(u, _reverb_taps(p, noise, 2 * fs), 0)
        else:
            pp = p.reshape(2, 20, 22)
            y = _conv(u, _Taps.apply(_zero_phase(pp[..., 2:], 39), pp[..., :2], int(round(0.1 * fs)), u.shape[-1]), -19)
        ey, eu = ((y[0] + y[1]) ** 2).sum(), ((u[0] + u[1]) ** 2).sum()
        lg = (0.5 * torch.log(ey + 1e-12) - 0.5 * torch.log(eu + 1e-12)).abs()
    return w * y + (1 - w) * u, lg


def _mel(nfft, fs):
    f = np.arange(nfft // 2 + 1) * fs / nfft
    top = 2595.0 * math.log10(1 + fs / 2 / 700.0)
    e = 700.0 * (10.0 ** (np.linspace(0, top, 98) / 2595.0) - 1)
    bank = np.stack([np.maximum(0.0, np.minimum((f - e[b]) / (e[b + 1] - e[b]), (e[b + 2] - f) / (e[b + 2] - e[b + 1]))) for b in range(96)])

    def ra(x):
        x = x * x
        return 12194.0 ** 2 * x * x / ((x + 20.6 ** 2) * np.sqrt((x + 107.7 ** 2) * (x + 737.9 ** 2)) * (x + 12194.0 ** 2))
    a = ra(f) / ra(np.float64(1000.0))
    return torch.as_tensor(bank, device="cuda"), torch.as_tensor(a, device="cuda")


def _audio_loss(case, mix, tgt):
    """(L_lr, L_m, L_s) of the multi-resolution STFT loss."""
    out = [torch.zeros((), dtype=D64, device="cuda") for _ in range(3)]
    for nfft in (case["fft0"], case["fft1"], case["fft2"]):
        hop = nfft // 4
        first = -(-case["warmup"] // hop)
        if mix.shape[1] < nfft or (mix.shape[1] - nfft) // hop + 1 <= first:
            continue
        bank, a = _mel(nfft, case["fs"])

        def spec(x):
            x = torch.stack([x[0], x[1], x[0] + x[1], x[0] - x[1]])
            z = torch.fft.rfft(x.unfold(1, nfft, hop)[:, first:] * _hann(nfft))
            return torch.sqrt(a ** 2 * (z.real ** 2 + z.imag ** 2) + 1e-8) @ bank.T
        y, x = spec(tgt.to(D64)), spec(mix)
        for i, sl in enumerate((slice(0, 2), slice(2, 3), slice(3, 4))):
            d = (torch.log(y[sl] + 1e-5) - torch.log(x[sl] + 1e-5)).abs().mean()
            out[i] = out[i] + d + torch.linalg.norm((y[sl] - x[sl]).reshape(-1)) / torch.linalg.norm(y[sl].reshape(-1))
    return out


def _exact_song(case, song, procs, src, tgt, noise, par, weight):
    """One song in 64 bits: losses [7], mix.  procs: (type, first parameter, processor, reverb) of its processors in
    order; weight(processor): its dry/wet weight."""
    k, s, group, n = song
    from torch.utils.checkpoint import checkpoint
    state = {"lg": torch.zeros((), dtype=D64, device="cuda")}
    it = iter(procs)

    def chain(u, steps):
        lg = torch.zeros((), dtype=D64, device="cuda")
        for t, o, q, rev in steps:
            u, l = _process(t, u, par[o:o + COUNT[t]], weight(q), noise[rev] if rev is not None else None, case["fs"])
            lg = lg + l
        return u, lg

    def run_chain(u, steps):
        if not steps:
            return u
        u, l = checkpoint(chain, u, steps, use_reentrant=False)
        state["lg"] = state["lg"] + l
        return u

    if case["graph"]:
        types, track, edges = _graph_of(case)
        out = {}
        for v, t in enumerate(types):
            if t == M.NODE_INPUT:
                out[v] = src[track[v]].to(D64).expand(2, n)
                continue
            u = sum(out[a] for a, b in sorted(edges) if b == v)
            out[v] = run_chain(u, [next(it)]) if t < 7 else u
        mix = out[len(types) - 1]
    else:
        per = len([t for t in ORDER if t in case["types"]])
        y = [run_chain(src[j].to(D64).expand(2, n), [next(it) for _ in range(per)]) for j in range(k)]
        mix = torch.zeros(2, n, dtype=D64, device="cuda")
        for g in range(s):
            u = torch.zeros(2, n, dtype=D64, device="cuda")
            for j in range(k):
                if group[j] == g:
                    u = u + y[j]
            mix = mix + run_chain(u, [next(it) for _ in range(per)])
        for j in range(k):
            if group[j] < 0:
                mix = mix + y[j]
    lr, m, sd = _audio_loss(case, mix, tgt)
    la = 0.5 * lr + 0.25 * m + 0.25 * sd
    lp = sum((weight(q) for _, _, q, _ in procs), torch.zeros((), dtype=D64, device="cuda"))
    total = la + 1e-3 * state["lg"] + ALPHA_P * lp
    return torch.stack([la, lr, m, sd, state["lg"], lp, total]), mix


def _metrics(est, ref, fs):
    """SI-SDR and the feature distances over 8 s segments."""
    a = (est * ref).sum() / (ref * ref).sum()
    sdr = 10 * torch.log10((a * ref).square().sum() / (a * ref - est).square().sum())
    n, seg = est.shape[1], int(round(8 * fs))
    parts = [(0, n)] if n < seg else [(i * seg, (i + 1) * seg) for i in range(n // seg)]
    edges = (0, 100, 200, 300, 400, 510, 630, 770, 920, 1080, 1270, 1480, 1720, 2000, 2320, 2700, 3150, 3700, 4400, 5300, 6400,
             7700, 9500, 12000, 15500)

    def feats(x):
        rms = x.square().mean(1).sqrt()
        l, r = x.square().sum(1)
        mid, c = (x[0] + x[1]) / 2, x.shape[1] // 8192
        f = torch.arange(4097, dtype=D64, device="cuda") * fs / 8192
        if c:
            pw = (torch.fft.rfft(mid[:c * 8192].reshape(c, 8192) * _hann(8192)).abs() ** 2).mean(0)
        else:
            pw = torch.zeros_like(f)
        bark = torch.stack([pw[(f >= edges[b]) & (f < edges[b + 1])].sum() for b in range(24)])
        return [rms, x.abs().amax(1) / rms, ((x[0] - x[1]).norm() / (x[0] + x[1]).norm())[None], ((l - r) / (l + r))[None],
                10 * torch.log10(bark + 1e-12)]
    acc = [[], [], [], [], []]
    for b, e in parts:
        for i, (p, q) in enumerate(zip(feats(est[:, b:e]), feats(ref[:, b:e]))):
            acc[i].append((p - q).square())
    return torch.stack([sdr] + [torch.log10(torch.cat(v).mean()) for v in acc])


def exact(case, seed):
    src, tgt, noise, params, masks, crop = _inputs(case, seed)
    songs, kind = _songs(case), case["kind"]
    where, o, rev = [], 0, 0
    for q, (t, i) in enumerate(_proc_types(case)):
        where.append((t, o, q, rev if t == "r" else None, i))
        o += COUNT[t]
        rev += t == "r"
    par = torch.as_tensor(params, dtype=D64, device="cuda").requires_grad_(kind not in ("score", "render"))
    losses, mixes, mets, las = [], [], [], []
    for i, song in enumerate(songs):
        n = song[3]
        a, b = src[i][:, crop:crop + n], tgt[i][:, crop:crop + n]
        mine = [w[:4] for w in where if w[4] == i]

        def one(mask):
            w = torch.sigmoid(par[o:])
            if mask is not None:
                w = w * torch.as_tensor(mask, dtype=D64, device="cuda")
            return _exact_song(case, song, mine, a, b, noise, par, lambda q: w[q])
        if kind == "score":
            with torch.no_grad():
                las.append(torch.stack([one(m)[0][0] for m in masks]))
            continue
        if kind == "render":
            with torch.no_grad():
                l, mix = one(masks)
                mets.append(_metrics(mix, b.to(D64), case["fs"]))
        else:
            l, mix = one(None)
            l[6].backward()
        losses.append(l.detach())
        mixes.append(mix.detach())
    if kind == "score":
        return {"la": torch.stack(las, 1)}
    if kind == "render":
        return {"losses": torch.stack(losses), "mix": mixes, "metrics": torch.stack(mets)}
    out = {"losses": torch.stack(losses), "grads": par.grad}
    if kind == "grad":
        out["mix"] = mixes
    return out
