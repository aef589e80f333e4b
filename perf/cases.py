"""The calls that a program using this library makes, over the range of sizes it makes them at.

Each case is one pass through a public entry point on FP32 signals (the
library's only signal type) with FP64 coefficient rows.  The filters are the
library's own workloads: Butterworth low-pass and band-pass designs, banks of
random sections (poles at radius 0.5..0.995, or 0.999..0.9999 for long
memories, zeros on the unit circle, unit peak gain) and Linkwitz-Riley
crossovers; signals and initial states are N(0, 1).  Lengths and section
counts of uneven batches come from the case's ``shape_seed``, everything else
from the seed given to ``prepare``.
"""
import math

import numpy as np
import torch

import paper_2607_14054_gb300 as P


def listed():
    return [
        # one short block of one channel, second-order low-pass: call latency
        {"name": "lowpass_8k", "kind": "single", "design": "lowpass", "K": 1, "length": 8192,
         "state": False},
        # live audio: 16 blocks of 256 samples on 16 channels, one call per block
        {"name": "stream_16x256", "kind": "stream", "K": 4, "channels": 16, "chunk": 256,
         "blocks": 16},
        # a recording of odd length continued from an earlier state
        {"name": "recording_1m", "kind": "single", "design": "bandpass", "K": 4,
         "length": 1_000_003, "state": True},
        # a long recording through a fourth-order band-pass: mostly memory traffic
        {"name": "bandpass4_32m", "kind": "single", "design": "bandpass", "K": 2,
         "length": 1 << 25, "state": False},
        # the headline: 16th-order band-pass of one long signal
        {"name": "bandpass16_16m", "kind": "single", "design": "bandpass", "K": 8,
         "length": 1 << 24, "state": False},
        # a service's batch: 4096 channels of uneven lengths and orders
        {"name": "batch_4096", "kind": "batch", "channels": 4096, "kmax": 8, "min_len": 1 << 10,
         "max_len": 1 << 20, "shape_seed": 3},
        # a data loader's batch of short clips, uneven lengths and orders
        {"name": "clips_1024", "kind": "batch", "channels": 1024, "kmax": 8, "min_len": 250,
         "max_len": 8200, "shape_seed": 4},
        # narrow resonators with memories of 1e4..1e5 samples, extended precision
        {"name": "resonators_64x4m", "kind": "resonators", "channels": 64, "K": 8,
         "length": 1 << 22},
        # a training step through a learnable filter layer: forward and all gradients
        {"name": "train_256x64k", "kind": "train", "channels": 256, "K": 8, "length": 1 << 16},
        # offline zero-phase filtering of a multi-channel recording
        {"name": "zerophase_64x100k", "kind": "zerophase", "channels": 64, "K": 4,
         "length": 100_003},
        # a loudspeaker crossover's low branch (coincident poles at a low cutoff)
        {"name": "crossover_16x100k", "kind": "crossover", "channels": 16, "length": 100_003,
         "wn": 0.002},
        # the headline filter on a signal in pinned host memory, result back in host memory
        {"name": "host_16m", "kind": "host", "design": "bandpass", "K": 8, "length": 1 << 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "stream", "batch", "batch", "resonators", "train",
                       "zerophase", "crossover", "host"])
    if kind == "single":
        K = rng.randint(1, 8)
        return {"kind": kind, "design": "lowpass" if K == 1 else "bandpass", "K": K,
                "length": _log_int(rng, 8192, 1 << 25), "state": rng.random() < 0.5}
    if kind == "stream":
        return {"kind": kind, "K": rng.randint(1, 8), "channels": _log_int(rng, 1, 64),
                "chunk": _log_int(rng, 64, 8192), "blocks": 16}
    if kind == "batch":
        longest = _log_int(rng, 8192, 1 << 18)
        return {"kind": kind, "channels": _log_int(rng, 16, 2048), "kmax": rng.randint(2, 8),
                "min_len": _log_int(rng, 250, 4000), "max_len": longest,
                "shape_seed": rng.randrange(1 << 20)}
    if kind == "resonators":
        return {"kind": kind, "channels": _log_int(rng, 8, 64), "K": rng.randint(2, 8),
                "length": _log_int(rng, 1 << 18, 1 << 22)}
    if kind == "train":
        return {"kind": kind, "channels": _log_int(rng, 8, 256), "K": rng.randint(1, 8),
                "length": _log_int(rng, 4000, 1 << 16)}
    if kind == "zerophase":
        return {"kind": kind, "channels": _log_int(rng, 1, 64), "K": rng.randint(1, 8),
                "length": _log_int(rng, 10_000, 400_000)}
    if kind == "crossover":
        return {"kind": kind, "channels": _log_int(rng, 1, 64),
                "length": _log_int(rng, 20_000, 400_000), "wn": rng.uniform(0.002, 0.005)}
    K = rng.randint(2, 8)
    return {"kind": kind, "design": "bandpass", "K": K, "length": _log_int(rng, 1 << 20, 1 << 24)}


# ---- filters ----------------------------------------------------------------

def _butter(design, K):
    """[K, 6] rows: low-pass of order 2K at 0.1, or band-pass 0.1..0.2 of order 2K."""
    order = 2 * K if design == "lowpass" else K
    proto = [complex(math.cos(t), math.sin(t)) for t in
             (math.pi * (2 * k + order + 1) / (2 * order) for k in range(order))]
    if design == "lowpass":
        W = math.tan(math.pi * 0.1 / 2)
        poles, zeros, wc = [p * W for p in proto], (1.0, 2.0, 1.0), 0.0
    else:
        o1, o2 = math.tan(math.pi * 0.1 / 2), math.tan(math.pi * 0.2 / 2)
        poles = []
        for p in proto:
            pb = p * (o2 - o1)
            d = (pb * pb - 4 * o1 * o2) ** 0.5
            poles += [(pb + d) / 2, (pb - d) / 2]
        zeros, wc = (1.0, 0.0, -1.0), 2 * math.atan(math.sqrt(o1 * o2))
    z = sorted(((1 + s) / (1 - s) for s in poles), key=abs)
    z = [p for p in z if p.imag > 0]
    rows = np.array([[*zeros, 1.0, -2 * p.real, abs(p) ** 2] for p in z])
    zi = complex(math.cos(wc), -math.sin(wc))
    h = 1.0
    for b0, b1, b2, _, a1, a2 in rows:
        h *= abs((b0 + b1 * zi + b2 * zi * zi) / (1 + a1 * zi + a2 * zi * zi))
    rows[:, :3] *= h ** (-1.0 / K)
    return rows


def _random_sections(r, n, rmin, rmax):
    """[n, 6] random sections of unit peak gain: |B|^2 / |A|^2 is a ratio of two
    quadratics in c = cos w, so its peak is at c = +-1 or at a root of a quadratic."""
    rad = r.uniform(rmin, rmax, n)
    th, ph = r.uniform(0, math.pi, n), r.uniform(0, math.pi, n)
    one = np.ones(n)
    b = np.stack([one, -2 * np.cos(ph), one], 1)
    a = np.stack([one, -2 * rad * np.cos(th), rad * rad], 1)

    def quadratic(p):  # |P|^2 = q0 + q1 c + q2 c^2
        q2 = 4 * p[:, 0] * p[:, 2]
        return (p * p).sum(1) - q2 / 2, 2 * p[:, 1] * (p[:, 0] + p[:, 2]), q2

    n0, n1, n2 = quadratic(b)
    d0, d1, d2 = quadratic(a)
    A, B, C = n2 * d1 - n1 * d2, 2 * (n2 * d0 - n0 * d2), n1 * d0 - n0 * d1
    disc = np.sqrt(np.maximum(B * B - 4 * A * C, 0))
    with np.errstate(divide="ignore", invalid="ignore"):
        roots = [(-B + disc) / (2 * A), (-B - disc) / (2 * A), -C / B]
    peak = np.zeros(n)
    for c in [one, -one] + [np.clip(np.nan_to_num(x, nan=1.0), -1, 1) for x in roots]:
        peak = np.maximum(peak, (n0 + n1 * c + n2 * c * c) / (d0 + d1 * c + d2 * c * c))
    return np.concatenate([b / np.sqrt(peak)[:, None], a], 1)


def _bank(r, C, kmax, K, rmin, rmax):
    rows = np.tile(np.array([1.0, 0, 0, 1, 0, 0]), (C, kmax, 1))  # past K: never read
    used = np.arange(kmax)[None, :] < np.asarray(K)[:, None]
    rows[used] = _random_sections(r, int(used.sum()), rmin, rmax)
    return rows


def _shape(case):
    """(lengths, K) of every channel."""
    kind = case["kind"]
    if kind == "batch":
        r = np.random.RandomState(case["shape_seed"])
        C = case["channels"]
        return (r.randint(case["min_len"], case["max_len"] + 1, C).tolist(),
                r.randint(1, case["kmax"] + 1, C).tolist())
    if kind in ("single", "host"):
        return [case["length"]], [case["K"]]
    if kind == "stream":
        return [case["chunk"] * case["blocks"]] * case["channels"], [case["K"]] * case["channels"]
    return [case["length"]] * case["channels"], [case.get("K", 2)] * case["channels"]


def _inputs(case, seed):
    """What the user holds: signal, rows, section counts, lengths, states."""
    lengths, K = _shape(case)
    C, kmax, kind = len(lengths), case.get("kmax", max(K)), case["kind"]
    r = np.random.RandomState(seed % (1 << 31))
    if kind in ("single", "host"):
        sos = _butter(case["design"], case["K"])[None]
    elif kind == "crossover":
        sos = np.tile(_butter_low2(case["wn"]), (C, 2, 1))
    elif kind == "resonators":
        sos = _bank(r, C, kmax, K, 0.999, 0.9999)
    else:
        sos = _bank(r, C, kmax, K, 0.5, 0.995)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(sum(lengths), device="cuda", generator=g)
    zi = None
    if kind in ("batch", "train") or case.get("state"):
        zi = torch.randn(C, kmax, 2, device="cuda", generator=g)
    gy = torch.randn(sum(lengths), device="cuda", generator=g) if kind == "train" else None
    return {"x": x, "sos": torch.from_numpy(sos).cuda(), "zi": zi, "gy": gy, "lengths": lengths,
            "K": torch.tensor(K, dtype=torch.int32, device="cuda"), "kmax": kmax}


def _butter_low2(wn):
    W = math.tan(math.pi * wn / 2)
    D = 1 + math.sqrt(2) * W + W * W
    g = W * W / D
    return np.array([[g, 2 * g, g, 1, 2 * (W * W - 1) / D, (1 - math.sqrt(2) * W + W * W) / D]])


# ---- the calls --------------------------------------------------------------

def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"] = kind = case["kind"]
    if kind in ("batch", "resonators"):
        s["plan"] = P.SosFilter(s["lengths"], s["kmax"])
    elif kind == "stream":
        s["stream"] = P.SosStream(s["sos"], case["chunk"])
        s["blocks"] = list(s["x"].view(case["blocks"], case["channels"], case["chunk"]))
    elif kind == "train":
        # the learnable rows are FP32 parameters, as an optimiser keeps them
        s["theta"] = s["sos"].float().requires_grad_(True)
        s["x"].requires_grad_(True)
        s["zi"].requires_grad_(True)
    elif kind == "host":
        s["x_host"] = s.pop("x").cpu().pin_memory()
        s["y_host"] = torch.empty_like(s["x_host"]).pin_memory()
    return s


def run(s):
    kind = s["kind"]
    if kind == "single":
        return P.sosfilt(s["x"], s["sos"], zi=s["zi"])
    if kind in ("batch", "resonators"):
        return s["plan"](s["x"], s["sos"], s["K"], s["zi"])
    if kind == "stream":
        s["stream"].reset()
        return [s["stream"](b) for b in s["blocks"]] + [s["stream"].state]
    if kind == "train":
        y, zf = P.sosfilt_diff(s["x"], s["theta"].double(), s["K"], lengths=s["lengths"],
                               zi=s["zi"])
        return (y, zf, *torch.autograd.grad(y, (s["x"], s["theta"], s["zi"]), s["gy"]))
    if kind == "zerophase":
        return P.sosfiltfilt(s["x"], s["sos"], s["K"], lengths=s["lengths"])
    if kind == "crossover":
        return P.sosfilt(s["x"], s["sos"], K=s["K"], lengths=s["lengths"])
    return P.sosfilt_host(s["x_host"], s["sos"], y_host=s["y_host"])


def work(case):
    """Each signal read once and written once, five multiply-adds per sample and
    section; a training step also reads dL/dy, writes dL/dx, and does the adjoint
    recursion (five) and the coefficient sums (five)."""
    lengths, K = _shape(case)
    n, nk = sum(lengths), sum(m * k for m, k in zip(lengths, K))
    kind = case["kind"]
    if kind == "train":
        return {"bytes": 16 * n, "flops": 2 * 15 * nk}
    return {"bytes": 8 * n, "flops": 2 * 5 * nk * (2 if kind == "zerophase" else 1)}


# ---- the same in 64 bits ----------------------------------------------------

def _section(x, row, z):
    """One section over x [C, T] from the transposed-direct-form-II state z [C, 2]: blocks
    run side by side from zero state, then each gets the response of its true state."""
    C, T = x.shape
    B = min(4096, 1 << max(5, (max(T, 1).bit_length() + 1) // 2))
    nb = -(-T // B)
    b0, b1, b2, a1, a2 = (row[:, i:i + 1] for i in range(5))
    # columns nb and nb + 1: the responses of the two unit states
    w = torch.zeros(B, C, nb + 2, dtype=torch.float64, device=x.device)
    w[:, :, :nb] = torch.nn.functional.pad(x, (0, nb * B - T)).view(C, nb, B).permute(2, 0, 1)
    s1, s2 = torch.zeros_like(w[0]), torch.zeros_like(w[0])
    s1[:, nb] = 1
    s2[:, nb + 1] = 1
    for u in w:
        y = torch.addcmul(s1, b0, u)
        s1 = torch.addcmul(torch.addcmul(s2, b1, u), a1, y, value=-1)
        s2 = torch.addcmul(b2 * u, a2, y, value=-1)
        u.copy_(y)
    end = torch.stack([s1, s2], 1)  # [C, 2, nb + 2]
    M, e = end[:, :, nb:].contiguous(), end[:, :, :nb].permute(2, 0, 1).unsqueeze(-1).contiguous()
    zs, v = [], z.unsqueeze(-1)
    for j in range(nb):
        zs.append(v)
        v = torch.baddbmm(e[j], M, v)
    zs = torch.cat(zs, 2)  # [C, 2, nb]
    w[:, :, :nb].addcmul_(w[:, :, nb:nb + 1].clone(), zs[:, 0])
    w[:, :, :nb].addcmul_(w[:, :, nb + 1:].clone(), zs[:, 1])
    return w[:, :, :nb].permute(1, 2, 0).reshape(C, nb * B)[:, :T]


def _last_state(x, y, row, z, n):
    """The section's state after n >= 2 samples, from its last inputs and outputs."""
    at = torch.stack([n - 1, n - 2], 1)
    u, v = x.gather(1, at), y.gather(1, at)
    _, b1, b2, a1, a2 = row.T
    return torch.stack([b1 * u[:, 0] + b2 * u[:, 1] - a1 * v[:, 0] - a2 * v[:, 1],
                        b2 * u[:, 0] - a2 * v[:, 0]], 1)


def _normalised(sos):
    return torch.cat([sos[..., :3], sos[..., 4:]], -1) / sos[..., 3:4]


def _cascade(x, rows, K, z, n, keep=False):
    """x [C, T] through rows [C, kmax, 5]; (output, final states, every section's output)."""
    C, kmax = rows.shape[:2]
    zf = torch.zeros(C, kmax, 2, dtype=torch.float64, device=x.device)
    signals = [x]
    for k in range(kmax):
        on = (K > k).nonzero().flatten()
        if on.numel() == 0:
            break
        whole = on.numel() == C
        u = x if whole else x[on]
        y = _section(u, rows[on, k], z[on, k])
        zf[on, k] = _last_state(u, y, rows[on, k], z[on, k], n[on])
        if whole:
            x = y
        else:
            x = x.clone()
            x[on] = y
        if keep:
            signals.append(x)
    return x, zf, signals


def exact(case, seed):
    s = _inputs(case, seed)
    kind, lengths = case["kind"], s["lengths"]
    sos = s["sos"].float().double() if kind == "train" else s["sos"]
    rows, K, C = _normalised(sos), s["K"], len(lengths)
    z = s["zi"].double() if s["zi"] is not None else torch.zeros(C, s["kmax"], 2,
                                                                 dtype=torch.float64, device="cuda")
    n = torch.tensor(lengths, device="cuda")
    if kind == "batch":
        y = torch.empty(sum(lengths), dtype=torch.float64, device="cuda")
        zf = torch.empty(C, s["kmax"], 2, dtype=torch.float64, device="cuda")
        off = np.concatenate([[0], np.cumsum(lengths)])
        order = np.argsort(lengths)
        for part in np.array_split(order, -(-C // 256)):
            x = torch.zeros(len(part), lengths[part[-1]], dtype=torch.float64, device="cuda")
            for i, c in enumerate(part):
                x[i, :lengths[c]] = s["x"][off[c]:off[c + 1]]
            at = torch.from_numpy(part).cuda()
            v, zf[at], _ = _cascade(x, rows[at], K[at], z[at], n[at])
            for i, c in enumerate(part):
                y[off[c]:off[c + 1]] = v[i, :lengths[c]]
        return y, zf
    if kind == "stream":
        x = s["x"].view(case["blocks"], C, case["chunk"]).double()
        y, zf, _ = _cascade(x.transpose(0, 1).reshape(C, -1), rows, K, z, n)
        return [b.contiguous() for b in y.reshape(C, case["blocks"], -1).unbind(1)] + [zf]
    x = s["x"].view(C, -1).double()
    if kind == "zerophase":
        y = _cascade(x, rows, K, z, n)[0].flip(1)
        return _cascade(y, rows, K, z, n)[0].flip(1).reshape(-1)
    y, zf, signals = _cascade(x, rows, K, z, n, keep=kind == "train")
    if kind != "train":
        return y.reshape(-1), zf
    g = s["gy"].view(C, -1).double()
    gsos, gzi = torch.zeros_like(sos), torch.zeros_like(z)
    for k in reversed(range(s["kmax"])):
        b, a = rows[:, k, :3], rows[:, k, 3:]
        # lambda_n = g_n - a1 lambda_{n+1} - a2 lambda_{n+2}: an all-pole section backwards
        pole = torch.cat([torch.tensor([[1.0, 0, 0]], device="cuda").double().expand(C, 3), a], 1)
        lam = _section(g.flip(1), pole, torch.zeros(C, 2, device="cuda").double()).flip(1)
        lam = torch.nn.functional.pad(lam, (0, 2))
        l0, l1, l2 = lam[:, :-2], lam[:, 1:-1], lam[:, 2:]
        u, v = signals[k], signals[k + 1]
        d = torch.stack([(l0 * u).sum(1), (l1 * u).sum(1), (l2 * u).sum(1), -(l1 * v).sum(1),
                         -(l2 * v).sum(1)], 1)
        a0 = sos[:, k, 3]
        gsos[:, k, :3], gsos[:, k, 4:] = d[:, :3] / a0[:, None], d[:, 3:] / a0[:, None]
        gsos[:, k, 3] = -(rows[:, k] * d).sum(1) / a0
        gzi[:, k] = lam[:, :2]
        g = b[:, :1] * l0 + b[:, 1:2] * l1 + b[:, 2:] * l2
    return y.reshape(-1), zf, g.reshape(-1), gsos, gzi
