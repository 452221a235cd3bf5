"""The work a correlator program has this library do, as timed cases.

Each case is one call, or one short sequence of calls, of the public binding
(``paper_1501_05992_gb300.corr``) at sizes an array of that kind runs:

* ``listed()``  the fixed cases;
* ``draw(rng)`` one more case of the same ranges;
* ``prepare(case, seed)`` the inputs, output buffers and contexts a program
  has in hand before the call; ``run(state)`` the call itself;
* ``work(case)`` the bytes and operations the result cannot do without;
* ``exact(case, seed)`` the result in plain 64-bit torch.

Voltages are 4+4-bit Gaussian noise of standard deviation 2.5 codes clipped
to +-7 (what a digitiser's gain control aims at), with a few code-8 bytes
(the format's "invalid" marker) where the case zeroes them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1501_05992_gb300 import corr

DEV = "cuda:0"
PIECE = 1 << 26                      # samples generated at a time


def listed():
    return [
        # the smallest call: a 16-input test array, one second of 32 channels
        dict(name="small_array", kind="integrate", n=16, f=32, t=1000, zero_invalid=False, n_avg=0),
        # one 1.28 MHz coarse channel of the 256-input array, half a second:
        # the share of the band one correlator node of 24 serves
        dict(name="coarse_channel", kind="integrate", n=256, f=128, t=5000, zero_invalid=False, n_avg=0),
        # the whole 30.72 MHz band of the 256-input array, half a second
        dict(name="full_band", kind="integrate", n=256, f=3072, t=5000, zero_invalid=False, n_avg=0),
        # an input count that is no multiple of 16, an odd length, invalid samples zeroed
        dict(name="ragged_array", kind="integrate", n=250, f=768, t=4990, zero_invalid=True, n_avg=0),
        # correlation and incoherent beam of the same samples (a quarter of the band)
        dict(name="with_beam", kind="integrate", n=256, f=768, t=5000, zero_invalid=False, n_avg=1),
        # the streaming service: three arrays, ten 50 ms blocks added as they arrive, then the dump
        dict(name="block_stream", kind="stream", arrays="256x768,128x768,512x768", block=500, blocks=10),
        # whole integrations of three arrays of uneven size in one call
        dict(name="uneven_batch", kind="batch", arrays="128x384x2000,256x768x5000,1024x128x10000"),
        # host buffers in, host triangle out: one coarse channel, half a second
        dict(name="host_stream", kind="host", n=256, f=128, t=5000),
        # one 50 ms bank of packets as the receiver collects them, a few lost or damaged
        dict(name="packet_bank", kind="ingest", bank=3, lost=0.001, damaged=0.0001),
        # archive order, averaged two by two in channel and dump (half the band)
        dict(name="remap_2x2", kind="remap", n=256, f=1536, f_avg=2, dumps=2),
        # the incoherent beam on its own, one 50 ms block at the voltage rate
        dict(name="beam_block", kind="beam", n=256, f=3072, t=500, n_avg=1, zero_invalid=False),
        # the fine filterbank of one 50 ms block, codes for the correlator
        dict(name="fine_pfb", kind="fpfb", q=24, n=256, frames=500, taps=12, spec=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["integrate", "integrate", "integrate", "stream", "batch", "host", "ingest", "remap", "beam",
                       "fpfb"])
    if kind == "integrate":
        n = rng.choice([_log_int(rng, 8, 1024), 16 * _log_int(rng, 1, 64), 128, 256, 512])
        t = _log_int(rng, 100, 10000)
        # the voltages, the triangle and the products stay within the listed ones' sizes
        cap = min(2e9 / (n * t), 4e8 / (8 * n * (n + 1) / 2), (4e11 if n >= 64 else 5e9) / (t * n * n / 2))
        f = max(1, _log_int(rng, 1, max(2, min(3072, int(cap)))))
        n_avg = rng.choice([0, 0, 0, 1, 10])
        if n_avg:
            t = max(1, t // n_avg) * n_avg
        return dict(kind=kind, n=n, f=f, t=t, zero_invalid=rng.random() < 0.3, n_avg=n_avg)
    if kind == "stream":
        ns = rng.sample([64, 128, 192, 256, 384, 512], rng.randint(1, 3))
        f = _log_int(rng, 24, 500)
        return dict(kind=kind, arrays=",".join(f"{n}x{f}" for n in ns), block=_log_int(rng, 100, 1000),
                    blocks=rng.randint(2, 10))
    if kind == "batch":
        ns = rng.sample([96, 128, 160, 256, 320, 512, 1024], rng.randint(2, 4))
        return dict(kind=kind, arrays=",".join(
            f"{n}x{_log_int(rng, 16, 60 if n > 512 else 300)}x{_log_int(rng, 300, 6000)}" for n in ns))
    if kind == "host":
        n = rng.choice([128, 256, 512])
        return dict(kind=kind, n=n, f=_log_int(rng, 16, 128), t=_log_int(rng, 400, 5000 if n < 512 else 2000))
    if kind == "ingest":
        return dict(kind=kind, bank=rng.randint(0, 19), lost=rng.choice([0.0, 0.001, 0.02]),
                    damaged=rng.choice([0.0, 0.0001]))
    if kind == "remap":
        n = rng.choice([64, 128, 256, 512])
        f_avg, dumps = rng.choice([(1, 1), (2, 2), (4, 1), (2, 1), (1, 3)])
        f = f_avg * _log_int(rng, 8, max(9, int(1500 * 256 ** 2 / n ** 2 / f_avg / dumps)))
        return dict(kind=kind, n=n, f=min(f, 3072 // f_avg * f_avg), f_avg=f_avg, dumps=dumps)
    if kind == "beam":
        n_avg = rng.choice([1, 5, 10])
        n = rng.choice([16 * rng.randint(2, 64), 128, 256, 512])
        t = n_avg * _log_int(rng, 20, 1000 // n_avg)
        return dict(kind=kind, n=n, f=_log_int(rng, 16, max(17, min(3072, int(4e8 / (n * t))))), t=t, n_avg=n_avg,
                    zero_invalid=rng.random() < 0.3)
    return dict(kind=kind, q=rng.choice([1, 2, 6, 12, 24]), n=rng.choice([16, 64, 100, 128, 256]),
                frames=_log_int(rng, 8, 500), taps=rng.choice([12, 12, 12, 1]), spec=rng.random() < 0.3)


# ------------------------------------------------------------------ inputs --

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 7919 * salt + 17)
    return g


def _voltages(shape, g, invalid=False):
    """uint8 bytes (real part in the high nibble) of Gaussian 4+4-bit samples."""
    out = torch.empty(shape, dtype=torch.uint8, device=DEV)
    flat = out.view(-1)
    for i in range(0, flat.numel(), PIECE):
        k = min(PIECE, flat.numel() - i)
        x = torch.randn((2, k), generator=g, device=DEV).mul_(2.5).round_().clamp_(-7, 7).to(torch.int8)
        b = ((x[0] << 4) | (x[1] & 15)).view(torch.uint8)
        if invalid:
            b = torch.where(torch.rand(k, generator=g, device=DEV) < 1e-3, torch.full_like(b, 0x88), b)
        flat[i:i + k] = b
    return out


def _arrays(case):
    return [tuple(int(x) for x in a.split("x")) for a in case["arrays"].split(",")]


def _tri(n, f):
    return torch.empty((f, n * (n + 1) // 2, 2), dtype=torch.int32, device=DEV)


def _window(taps):
    """One-channel-wide Kaiser-windowed sinc of taps x 128 samples, summing to 128."""
    if taps == 1:
        return np.ones(128)
    x = np.arange(taps * 128)
    c = (taps * 128 - 1) / 2
    w = np.kaiser(taps * 128, 5.0) * np.sinc((x - c) / 128)
    return w * 128 / w.sum()


def _pfb_inputs(case, seed):
    g = _gen(seed)
    s = 128 * (case["frames"] + case["taps"] - 1)
    x = torch.empty((case["q"], case["n"], s, 2), dtype=torch.int8, device=DEV)
    for q in range(case["q"]):
        x[q] = torch.randn(x.shape[1:], generator=g, device=DEV).mul_(8).round_().clamp_(-127, 127).to(torch.int8)
    win = _window(case["taps"])
    scale = 2.5 / (8 * math.sqrt(float((win ** 2).sum())))    # white noise to 2.5 codes
    return x, torch.from_numpy(win.astype(np.float32)).to(DEV), scale


def _bank(case, seed):
    """A bank's voltage block and its packets in arrival order: for each coarse
    channel the 32 lanes' blocks of 2000 packets (4 groups x 500 frames)."""
    g = _gen(seed)
    block = _voltages((500, 3072, 256), g)
    # [frame][c][mgt][grp][f2][pfb][k] -> [c][pfb][mgt][grp][frame][f2][k]
    data = block.view(500, 24, 8, 4, 4, 4, 64).permute(1, 5, 2, 3, 0, 4, 6).reshape(-1, 256)
    pk = torch.empty((data.shape[0], 264), dtype=torch.uint8, device=DEV)
    pk[:, 6:262] = data
    idx = torch.arange(data.shape[0], device=DEV)
    frame, grp, mgt = idx % 500, idx // 500 % 4, idx // 2000 % 8
    pfb, chan = idx // 16000 % 4, idx // 64000
    tick = ((case["bank"] == 0) & (chan == 0) & (grp == 0) & (frame == 0)).long()
    w2 = tick | (pfb << 4) | (mgt << 6) | (case["bank"] << 9)
    w3 = frame | (grp << 9) | (chan << 11)
    pk[:, 0], pk[:, 1] = 0x08, 0x00
    pk[:, 2], pk[:, 3] = (w2 >> 8).to(torch.uint8), (w2 & 255).to(torch.uint8)
    pk[:, 4], pk[:, 5] = (w3 >> 8).to(torch.uint8), (w3 & 255).to(torch.uint8)
    x = data.view(-1, 128, 2)
    n = 128
    while n > 1:
        n //= 2
        x = x[:, :n] ^ x[:, n:2 * n]
    pk[:, 262:264] = x[:, 0]
    bad = torch.rand(data.shape[0], generator=g, device=DEV) < case["damaged"]
    lost = torch.rand(data.shape[0], generator=g, device=DEV) < case["lost"]
    pk[:, 100] ^= bad.to(torch.uint8)
    return block, pk[~lost].contiguous(), lost, bad


# ---------------------------------------------------------- prepare and run --

def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "integrate":
        n, f, t = case["n"], case["f"], case["t"]
        s["c"] = corr.Correlator(n, f, t, zero_invalid=case["zero_invalid"])
        s["volt"] = _voltages((t, f, n), _gen(seed), case["zero_invalid"])
        s["out"] = _tri(n, f)
        if case["n_avg"]:
            s["beam"] = torch.empty((t // case["n_avg"], f), dtype=torch.int32, device=DEV)
    elif kind == "stream":
        arrays = _arrays(case)
        s["b"] = corr.Batch([(n, f, case["block"] * case["blocks"]) for n, f in arrays])
        # a ring of three device slots per array, as the service keeps
        s["ring"] = [[_voltages((case["block"], f, n), _gen(seed, 10 * a + k)) for a, (n, f) in enumerate(arrays)]
                     for k in range(3)]
        s["outs"] = [_tri(n, f) for n, f in arrays]
    elif kind == "batch":
        arrays = _arrays(case)
        s["b"] = corr.Batch(arrays)
        s["volts"] = [_voltages((t, f, n), _gen(seed, a)) for a, (n, f, t) in enumerate(arrays)]
        s["outs"] = [_tri(n, f) for n, f, _ in arrays]
    elif kind == "host":
        n, f, t = case["n"], case["f"], case["t"]
        s["c"] = corr.Correlator(n, f, t)
        s["volt"] = _voltages((t, f, n), _gen(seed)).cpu().pin_memory()
        s["out"] = torch.empty((f, n * (n + 1) // 2, 2), dtype=torch.int32, pin_memory=True)
    elif kind == "ingest":
        s["pk"] = _bank(case, seed)[1]
        s["volt"] = torch.empty((500, 3072, 256), dtype=torch.uint8, device=DEV)
        s["seen"] = torch.empty(corr.PKT_SLOTS, dtype=torch.uint8, device=DEV)
        s["counters"] = torch.empty(corr.PKT_COUNTERS, dtype=torch.int32, device=DEV)
    elif kind == "remap":
        n, f = case["n"], case["f"]
        g = _gen(seed)
        s["tris"] = [torch.randint(-(1 << 17), 1 << 17, (f, n * (n + 1) // 2, 2), generator=g, device=DEV,
                                   dtype=torch.int32) for _ in range(case["dumps"])]
        st = n // 2
        s["out"] = torch.empty((f // case["f_avg"], st * (st + 1) // 2, 2, 2, 2), dtype=torch.int32, device=DEV)
    elif kind == "beam":
        s["volt"] = _voltages((case["t"], case["f"], case["n"]), _gen(seed), case["zero_invalid"])
        s["out"] = torch.empty((case["t"] // case["n_avg"], case["f"]), dtype=torch.int32, device=DEV)
    else:
        s["x"], s["win"], s["scale"] = _pfb_inputs(case, seed)
        shape = (case["frames"], case["q"] * 128, case["n"])
        s["volt"] = torch.empty(shape, dtype=torch.uint8, device=DEV)
        s["spec"] = torch.empty(shape + (2,), dtype=torch.float32, device=DEV) if case["spec"] else False
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "integrate":
        if case["n_avg"]:
            return list(s["c"].integrate_beam(s["volt"], case["n_avg"], out=s["out"], beam=s["beam"]))
        return [s["c"].integrate(s["volt"], out=s["out"])]
    if kind == "stream":
        for k in range(case["blocks"]):
            s["b"].accumulate(s["ring"][k % 3])
        return list(s["b"].dump(s["outs"]))
    if kind == "batch":
        return list(s["b"].integrate(s["volts"], s["outs"]))
    if kind == "host":
        s["c"].accumulate_host(s["volt"])
        return [s["c"].dump_host(s["out"])]
    if kind == "ingest":
        return list(corr.ingest_packets(s["pk"], case["bank"], out=s["volt"], seen=s["seen"],
                                        counters=s["counters"]))
    if kind == "remap":
        return [corr.remap(s["tris"], None, case["f_avg"], out=s["out"])]
    if kind == "beam":
        return [corr.incoherent_beam(s["volt"], case["n_avg"], case["zero_invalid"], out=s["out"])]
    volt, spec = corr.fine_pfb(s["x"], s["win"], s["scale"], volt=s["volt"], spec=s["spec"])
    return [volt, spec] if case["spec"] else [volt]


# -------------------------------------------------------------- work, exact --

def work(case):
    kind = case["kind"]

    def x_work(n, f, t):
        pairs = n * (n + 1) // 2
        return n * f * t + 8 * pairs * f, 8 * pairs * f * t

    if kind in ("integrate", "host"):
        b, ops = x_work(case["n"], case["f"], case["t"])
        if case.get("n_avg"):
            b += 4 * case["f"] * (case["t"] // case["n_avg"])
            ops += 4 * case["n"] * case["f"] * case["t"]
    elif kind in ("stream", "batch"):
        b = ops = 0
        for a in _arrays(case):
            w = x_work(a[0], a[1], a[2] if kind == "batch" else case["block"] * case["blocks"])
            b, ops = b + w[0], ops + w[1]
    elif kind == "ingest":
        b, ops = int(264 * 1536000 * (1 - case["lost"])) + 500 * 3072 * 256, 0
    elif kind == "remap":
        n, st = case["n"], case["n"] // 2
        b = case["dumps"] * case["f"] * n * (n + 1) * 4 + case["f"] // case["f_avg"] * st * (st + 1) * 16
        ops = case["dumps"] * case["f"] * n * (n + 1)
    elif kind == "beam":
        b = case["n"] * case["f"] * case["t"] + 4 * case["f"] * (case["t"] // case["n_avg"])
        ops = 4 * case["n"] * case["f"] * case["t"]
    else:
        per = case["q"] * case["n"] * case["frames"]
        b = per * 128 * (9 if case["spec"] else 1) + case["q"] * case["n"] * 256 * (case["frames"] + case["taps"] - 1)
        ops = per * (128 * 4 * case["taps"] + 5 * 128 * 7)
    return {"bytes": int(b), "flops": int(ops)}


def _parts(volt, zero_invalid):
    """Real and imaginary parts of packed bytes, as float64."""
    v = volt.view(torch.int8)
    r, m = v >> 4, (v << 4) >> 4
    if zero_invalid:
        bad = (r == -8) | (m == -8)
        r, m = r.masked_fill(bad, 0), m.masked_fill(bad, 0)
    return r.double(), m.double()


def _triangle(volt, zero_invalid=False):
    """int32 [F][P][2] of uint8 [T][F][N], sums in float64."""
    t, f, n = volt.shape
    i, j = torch.tril_indices(n, n, device=volt.device)
    out = _tri(n, f)
    step = max(1, (1 << 27) // (t * n))
    for f0 in range(0, f, step):
        r, m = _parts(volt[:, f0:f0 + step].permute(1, 2, 0).contiguous(), zero_invalid)
        rt, mt = r.transpose(1, 2), m.transpose(1, 2)
        out[f0:f0 + step, :, 0] = (r @ rt + m @ mt)[:, i, j].to(torch.int32)
        out[f0:f0 + step, :, 1] = (m @ rt - r @ mt)[:, i, j].to(torch.int32)
    return out


def _beam(volt, n_avg, zero_invalid):
    t, f, n = volt.shape
    out = torch.empty((t, f), dtype=torch.float64, device=volt.device)
    step = max(1, (1 << 26) // (f * n))
    for t0 in range(0, t, step):
        r, m = _parts(volt[t0:t0 + step], zero_invalid)
        out[t0:t0 + step] = (r * r + m * m).sum(-1)
    return out.view(t // n_avg, n_avg, f).sum(1).to(torch.int32)


def exact(case, seed):
    kind = case["kind"]
    if work(case)["flops"] > 2e12:
        return None                                  # more than a few seconds of 64-bit arithmetic
    if kind in ("integrate", "host"):
        zi = case.get("zero_invalid", False)
        volt = _voltages((case["t"], case["f"], case["n"]), _gen(seed), zi)
        out = [_triangle(volt, zi)]
        if case.get("n_avg"):
            out.append(_beam(volt, case["n_avg"], zi))
        return [o.cpu() for o in out] if kind == "host" else out
    if kind == "stream":
        out = []
        for a, (n, f) in enumerate(_arrays(case)):
            tris = [_triangle(_voltages((case["block"], f, n), _gen(seed, 10 * a + k))) for k in range(3)]
            out.append(sum(tris[k % 3] for k in range(case["blocks"])))
        return out
    if kind == "batch":
        return [_triangle(_voltages((t, f, n), _gen(seed, a))) for a, (n, f, t) in enumerate(_arrays(case))]
    if kind == "ingest":
        block, pk, lost, bad = _bank(case, seed)
        gone = (lost | bad).view(24, 4, 8, 4, 500).permute(4, 0, 2, 3, 1)          # [frame][c][mgt][grp][pfb]
        v = block.view(500, 24, 8, 4, 4, 4, 64)
        v.masked_fill_(gone[:, :, :, :, None, :, None], 0x88)
        n_bad = int((bad & ~lost).sum())
        counters = torch.tensor([pk.shape[0] - n_bad, 0, n_bad, 0, 0, int((lost | bad).sum())], dtype=torch.int32,
                                device=DEV)
        return [block, counters]
    if kind == "remap":
        n, f = case["n"], case["f"]
        tot = sum(t.long() for t in prepare(case, seed)["tris"]).view(f // case["f_avg"], case["f_avg"], -1, 2).sum(1)
        i, j = torch.tril_indices(n, n, device=DEV)
        pos = torch.arange(n, device=DEV)
        k = pos % 64
        nat = pos // 64 * 64 + k % 4 * 16 + k // 4
        full = torch.empty((tot.shape[0], n, n, 2), dtype=torch.int32, device=DEV)
        conj = torch.tensor([1, -1], device=DEV)
        full[:, nat[j], nat[i]] = (tot * conj).to(torch.int32)
        full[:, nat[i], nat[j]] = tot.to(torch.int32)
        a, b = torch.tril_indices(n // 2, n // 2, device=DEV)
        return [full.view(-1, n // 2, 2, n // 2, 2, 2)[:, a, :, b].transpose(0, 1).contiguous()]
    if kind == "beam":
        volt = _voltages((case["t"], case["f"], case["n"]), _gen(seed), case["zero_invalid"])
        return [_beam(volt, case["n_avg"], case["zero_invalid"])]
    if not case["spec"]:
        return None                                  # codes alone: bytes, rounded from the spectra
    x, _, _ = _pfb_inputs(case, seed)
    # the window a program hands over is float32; its values in 64 bits
    win = torch.from_numpy(_window(case["taps"]).astype(np.float32)).to(DEV).double().view(case["taps"], 128)
    m = case["frames"]
    spec = torch.empty((m, case["q"], 128, case["n"], 2), dtype=torch.float64, device=DEV)
    for q in range(case["q"]):
        for i in range(case["n"]):
            z = torch.view_as_complex(x[q, i].double()).view(-1, 128)
            u = sum(z[p:p + m] * win[p] for p in range(case["taps"]))
            spec[:, q, :, i] = torch.view_as_real(torch.fft.fft(u, dim=1).roll(64, dims=1))
    return [None, spec.view(m, case["q"] * 128, case["n"], 2)]
