"""The correlator's workloads as measurable cases, each a call sequence of a user's program.

A case is a dict of plain values. `kind` names the call sequence:

* xengine   one integration of an array: accumulate one block (or a batch of `blocks` resident blocks) of
            `n_time` samples, dump the visibilities and the total power, both restarted. `fmt` is the dump
            format. With `outriggers` > 0 the total power is dumped for that many stations only, the
            selective dump that runs beside the cross-power cadence.
* group     several sub-arrays (`arrays`, "inputs x channels" separated by commas) correlated by one grouped
            launch, then dumped.
* autos     the total-power cadence on its own: accumulate the autocorrelations of one block and dump them.
* requant   the F-engine's tail: gain, 4+4-bit requantisation, channel selection and corner turn.
* pfb       the F-engine's polyphase filterbank, 8192-point, `n_taps` taps.
* turn      the two local halves of the corner turn across processors: one board's spectra cut into the
            blocks of `n_dest` processors, and the blocks of `n_src` boards merged for one processor.

Sample values are receiver noise (sigma 2.5 in units of the 4-bit step) with a common signal of a tenth of
the power in every input, clipped to [-8, 7], as the requantiser hands them over.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1411_3751_gb300 import corr, replicas

FMT = {"ci64": corr.CORR_FMT_CI64, "cf32": corr.CORR_FMT_CF32, "cf32_norm": corr.CORR_FMT_CF32_NORM}
M = 8192           # PFB points
F = M // 2         # PFB channels
MAX_CMAC = 2.21e12     # the largest listed integration: complex products, input bytes, output cells
MAX_IN_BYTES = 8.7e9
MAX_OUT_BYTES = 1.2e9


def _xe(name, n, c, t, blocks=1, npol=2, fmt="ci64", outriggers=0):
    return {"name": name, "kind": "xengine", "n_inputs": n, "n_chans": c, "n_time": t, "blocks": blocks, "n_pol": npol,
            "fmt": fmt, "outriggers": outriggers}


def listed():
    return [
        # the smallest call: 16 dual-polarisation stations, a few channels, one short block (latency, launches)
        _xe("tiny_32x8x1024", 32, 8, 1024),
        # a 64-input station array's stream: one gulp of 25 blocks of 10 ms, full band
        _xe("lwa_64x2400x6000", 64, 2400, 6000, fmt="cf32"),
        # a small array with its blocks resident, one batch
        _xe("small_32x2400x4x8192", 32, 2400, 8192, blocks=4),
        # a mid-size array whose rows are not multiples of 16 bytes
        _xe("mid_200x300x4096", 200, 300, 4096, fmt="cf32"),
        # odd sizes: single polarisation, ragged inputs, channels and samples, a short batch
        _xe("ragged_131x109x1001", 131, 109, 1001, blocks=3, npol=1, fmt="cf32_norm"),
        # one processor's 109 channels of the 512-input array at the minimum dump time: one group of 8000
        # spectra, averaged visibilities, total power of ten outrigger stations
        _xe("leda_512x109x8000", 512, 109, 8000, fmt="cf32_norm", outriggers=10),
        # the benchmark's integration: 512 inputs, 128 channels, 16 blocks of 8192 samples
        _xe("leda_512x128x16x8192", 512, 128, 8192, blocks=16),
        # five uneven sub-arrays in one grouped launch
        {"name": "group_five_4096", "kind": "group", "arrays": "32x2400,64x600,200x300,256x150,512x109", "n_time": 4096,
         "n_pol": 2, "fmt": "ci64"},
        # total power of the full band every 10 ms
        {"name": "power_512x2400x240", "kind": "autos", "n_inputs": 512, "n_chans": 2400, "n_time": 240, "n_pol": 2,
         "fmt": "cf32"},
        # the F-engine's tail at full array and band: 18+18-bit integers in, 2398 of 4096 channels out
        {"name": "requant_512x256x2398", "kind": "requant", "n_inputs": 512, "n_time": 256, "chan0": 1229, "n_chans": 2398,
         "in_type": "int32", "gains": False, "symmetric": False},
        # the F-engine's filterbank at full array
        {"name": "pfb_512x64", "kind": "pfb", "n_inputs": 512, "n_spectra": 64, "n_taps": 4},
        # 16 boards of 32 inputs to 22 processors of 109 channels
        {"name": "turn_16x32_to_22x109", "kind": "turn", "n_src": 16, "n_local": 32, "n_dest": 22, "n_chans": 2398,
         "n_time": 1000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fits(n, c, t, blocks, npol):
    cells = (n // npol) * (n // npol + 1) // 2 * npol * npol * c
    return (n * (n + 1) / 2 * c * t * blocks <= MAX_CMAC and n * c * t * blocks <= MAX_IN_BYTES
            and cells * 16 <= MAX_OUT_BYTES)


def draw(rng):
    kind = rng.choice(["xengine"] * 6 + ["group", "autos", "requant", "pfb", "turn"])
    if kind == "xengine":
        while True:
            n = _log(rng, 2, 768)
            if rng.random() < 0.6:  # most arrays are built of boards of 16 inputs
                n = max(16, n // 16 * 16)
            npol = 1 if n % 2 or rng.random() < 0.2 else 2
            c, t, blocks = _log(rng, 1, 2400), _log(rng, 64, 16384), rng.choice([1, 1, 2, 3, 4, 7, 16])
            if rng.random() < 0.4:
                t = max(128, t // 128 * 128)
            if _fits(n, c, t, blocks, npol):
                break
        case = _xe("", n, c, t, blocks, npol, rng.choice(sorted(FMT)), rng.choice([0, 0, 0, min(10, n // npol)]))
        del case["name"]
        return case
    if kind == "group":
        shapes = []
        t = _log(rng, 256, 8192)
        while len(shapes) < 2 or (len(shapes) < 6 and rng.random() < 0.6):
            n, c = 2 * _log(rng, 4, 256), _log(rng, 4, 2400)
            if rng.random() < 0.6:
                n = max(16, n // 16 * 16)
            if _fits(n, c, t, 6, 2):
                shapes.append("%dx%d" % (n, c))
        return {"kind": "group", "arrays": ",".join(shapes), "n_time": t, "n_pol": 2, "fmt": rng.choice(sorted(FMT))}
    if kind == "autos":
        n = _log(rng, 2, 768)
        npol = 1 if n % 2 else 2
        c = _log(rng, 8, 2400)
        t = _log(rng, 64, min(16384, int(MAX_IN_BYTES // (n * c))))
        return {"kind": "autos", "n_inputs": n, "n_chans": c, "n_time": t, "n_pol": npol, "fmt": rng.choice(sorted(FMT))}
    if kind == "requant":
        n, t = _log(rng, 8, 512), _log(rng, 8, 256)
        c = _log(rng, 100, 2400)
        return {"kind": "requant", "n_inputs": n, "n_time": t, "chan0": rng.randrange(0, F - c), "n_chans": c,
                "in_type": rng.choice(["int32", "float32"]), "gains": rng.random() < 0.5, "symmetric": rng.random() < 0.5}
    if kind == "pfb":
        return {"kind": "pfb", "n_inputs": _log(rng, 2, 512), "n_spectra": _log(rng, 1, 64),
                "n_taps": rng.choice([4, 4, 4, 1, 2, 3, 8])}
    n_src, n_local = rng.randint(1, 16), rng.choice([16, 32, 32, 32, 12, 10])
    n_dest = rng.randint(1, 22)
    return {"kind": "turn", "n_src": n_src, "n_local": n_local, "n_dest": n_dest,
            "n_chans": rng.randint(max(32, n_dest), 2398), "n_time": _log(rng, 16, 1000)}


# ---- inputs ---------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _samples(g, t, c, n):
    """uint8 [t][c][n] packed 4+4-bit samples."""
    out = torch.empty((t, c, n), dtype=torch.uint8, device="cuda")
    step = max(1, (1 << 26) // (c * n))
    sigma, rho = 2.5, 0.1

    def part(m):
        noise = torch.randn((m, c, n), device="cuda", generator=g).mul_(sigma * math.sqrt(1.0 - rho))
        common = torch.randn((m, c, 1), device="cuda", generator=g).mul_(sigma * math.sqrt(rho))
        return noise.add_(common).round_().clamp_(-8, 7).to(torch.int8)

    for t0 in range(0, t, step):
        m = min(step, t - t0)
        re, im = part(m), part(m)
        out[t0:t0 + m] = ((re << 4) | (im & 15)).view(torch.uint8)
    return out


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["arrays"].split(",")]


def _stations(case):
    """The outrigger stations: spread over the array, the last ones first."""
    s = case["n_inputs"] // case["n_pol"]
    k = case["outriggers"]
    return [s - 1 - (i * s) // k for i in range(k)]


def _blocks(case, seed):
    g = _generator(seed)
    return [_samples(g, case["n_time"], case["n_chans"], case["n_inputs"]) for _ in range(case.get("blocks", 1))]


def _pfb_input(case, seed):
    g = _generator(seed)
    n, s = case["n_inputs"], (case["n_spectra"] + case["n_taps"] - 1) * M
    adc = torch.empty((n, s), dtype=torch.int8, device="cuda")
    tone = torch.cos(torch.arange(s, device="cuda", dtype=torch.float32) * (2.0 * math.pi * 0.1372)).mul_(6.0)
    for i in range(0, n, 16):
        x = torch.randn((min(16, n - i), s), device="cuda", generator=g).mul_(20.0).add_(tone)
        adc[i:i + 16] = x.round_().clamp_(-128, 127).to(torch.int8)
    return adc


def _requant_input(case, seed):
    g = _generator(seed)
    n, t = case["n_inputs"], case["n_time"]
    int32 = case["in_type"] == "int32"
    x = torch.empty((n, t, F, 2), dtype=torch.int32 if int32 else torch.float32, device="cuda")
    for i in range(0, n, 16):
        v = torch.randn((min(16, n - i), t, F, 2), device="cuda", generator=g).mul_(3000.0)
        x[i:i + 16] = v.round_().clamp_(-(1 << 17), (1 << 17) - 1).to(torch.int32) if int32 else v
    gains = None
    if case["gains"]:
        gains = torch.rand((case["n_chans"],), device="cuda", generator=g).mul_(1.0e-3).add_(4.0e-4)
    return x, gains


def _empty_dumps(xc, fmt, outriggers):
    dtype = torch.int64 if fmt == "ci64" else torch.float32
    autos = xc.station_out_shape(corr.CORR_WHAT_AUTO, outriggers) if outriggers else xc.out_shape(corr.CORR_WHAT_AUTO)
    return (torch.empty(xc.out_shape(corr.CORR_WHAT_CROSS), dtype=dtype, device="cuda"),
            torch.empty(autos, dtype=dtype, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "xengine":
        st["blocks"] = _blocks(case, seed)
        st["xc"] = corr.Correlator(case["n_inputs"], case["n_chans"], case["n_time"], case["n_pol"])
        st["cross"], st["autos"] = _empty_dumps(st["xc"], case["fmt"], case["outriggers"])
        st["stations"] = _stations(case)
    elif kind == "group":
        g = _generator(seed)
        shapes = _shapes(case)
        st["blocks"] = [_samples(g, case["n_time"], c, n) for n, c in shapes]
        st["group"] = corr.Group(shapes, case["n_time"], case["n_pol"])
        st["out"] = [_empty_dumps(m, case["fmt"], 0) for m in st["group"].members]
    elif kind == "autos":
        st["block"] = _blocks(case, seed)[0]
        st["xc"] = corr.Correlator(case["n_inputs"], case["n_chans"], case["n_time"], case["n_pol"])
        st["autos"] = torch.empty(st["xc"].out_shape(corr.CORR_WHAT_AUTO),
                                  dtype=torch.int64 if case["fmt"] == "ci64" else torch.float32, device="cuda")
    elif kind == "requant":
        st["x"], st["gains"] = _requant_input(case, seed)
        st["out"] = torch.empty((case["n_time"], case["n_chans"], case["n_inputs"]), dtype=torch.uint8, device="cuda")
    elif kind == "pfb":
        st["adc"] = _pfb_input(case, seed)
        st["out"] = torch.empty((case["n_inputs"], case["n_spectra"], F, 2), dtype=torch.float32, device="cuda")
    else:
        g = _generator(seed)
        n = case["n_src"] * case["n_local"]
        chan_b = [r[0] for r in replicas.channel_shards(case["n_chans"], case["n_dest"])] + [case["n_chans"]]
        own = chan_b[1]  # the first processor's channels
        st["board"] = _samples(g, case["n_time"], case["n_chans"], case["n_local"])
        st["received"] = _samples(g, case["n_time"], own, n).view(-1)
        st["packed"] = torch.empty((case["n_time"] * case["n_chans"] * case["n_local"],), dtype=torch.uint8, device="cuda")
        st["turned"] = torch.empty((case["n_time"], own, n), dtype=torch.uint8, device="cuda")
        st["chan_bounds"] = chan_b
        st["input_bounds"] = [case["n_local"] * i for i in range(case["n_src"] + 1)]
    return st


# ---- one pass -------------------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "xengine":
        xc = st["xc"]
        if len(st["blocks"]) == 1:
            xc.accumulate(st["blocks"][0])
        else:
            xc.accumulate_batch(st["blocks"])
        xc.dump(corr.CORR_WHAT_CROSS, FMT[case["fmt"]], reset=True, out=st["cross"])
        if st["stations"]:
            xc.dump_stations(st["stations"], corr.CORR_WHAT_AUTO, FMT[case["fmt"]], reset=True, out=st["autos"])
        else:
            xc.dump(corr.CORR_WHAT_AUTO, FMT[case["fmt"]], reset=True, out=st["autos"])
        return {"cross": st["cross"], "autos": st["autos"]}
    if kind == "group":
        st["group"].accumulate(st["blocks"])
        for m, (cross, autos) in zip(st["group"].members, st["out"]):
            m.dump(corr.CORR_WHAT_CROSS, FMT[case["fmt"]], reset=True, out=cross)
            m.dump(corr.CORR_WHAT_AUTO, FMT[case["fmt"]], reset=True, out=autos)
        return [{"cross": c, "autos": a} for c, a in st["out"]]
    if kind == "autos":
        st["xc"].accumulate_autos(st["block"])
        st["xc"].dump(corr.CORR_WHAT_AUTO, FMT[case["fmt"]], reset=True, out=st["autos"])
        return {"autos": st["autos"]}
    if kind == "requant":
        return corr.requantize(st["x"], case["chan0"], case["n_chans"], gain=8.0e-4, gains=st["gains"],
                               symmetric=case["symmetric"], out=st["out"])
    if kind == "pfb":
        return corr.pfb(st["adc"], case["n_taps"], out=st["out"])
    stream = torch.cuda.current_stream().cuda_stream
    corr.corr_corner_turn_pack(st["board"].data_ptr(), case["n_time"], case["n_chans"], case["n_local"], st["chan_bounds"],
                               st["packed"].data_ptr(), stream)
    corr.corr_corner_turn_unpack(st["received"].data_ptr(), case["n_time"], st["turned"].shape[1], st["turned"].shape[2],
                                 st["input_bounds"], st["turned"].data_ptr(), stream)
    return {"packed": st["packed"], "turned": st["turned"]}


# ---- what a pass cannot do without ----------------------------------------------------------------
def _xe_work(n, c, t, npol, fmt, outriggers=0):
    esz = 8 if fmt == "ci64" else 4
    s = n // npol
    cross = c * (s * (s + 1) // 2) * npol * npol * 2 * esz
    autos = c * (outriggers * npol if outriggers else n) * esz
    return n * c * t + cross + autos, 8.0 * (n * (n + 1) // 2) * c * t


def work(case):
    kind = case["kind"]
    if kind == "xengine":
        b, f = _xe_work(case["n_inputs"], case["n_chans"], case["n_time"] * case["blocks"], case["n_pol"], case["fmt"],
                        case["outriggers"])
        return {"bytes": b, "flops": f}
    if kind == "group":
        parts = [_xe_work(n, c, case["n_time"], case["n_pol"], case["fmt"]) for n, c in _shapes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind == "autos":
        cells = case["n_inputs"] * case["n_chans"]
        return {"bytes": cells * case["n_time"] + cells * (8 if case["fmt"] == "ci64" else 4),
                "flops": 4.0 * cells * case["n_time"]}
    if kind == "requant":
        s = case["n_inputs"] * case["n_time"] * case["n_chans"]
        return {"bytes": 9 * s + (4 * case["n_chans"] if case["gains"] else 0), "flops": 2.0 * s}
    if kind == "pfb":
        spectra = case["n_inputs"] * case["n_spectra"]
        frames = case["n_inputs"] * (case["n_spectra"] + case["n_taps"] - 1)
        return {"bytes": frames * M + spectra * F * 8 + 4 * M * case["n_taps"],
                "flops": spectra * (2.0 * case["n_taps"] * M + 5.0 * F * math.log2(F) + 10.0 * F)}
    own = replicas.channel_shards(case["n_chans"], case["n_dest"])[0]
    moved = case["n_time"] * (case["n_chans"] * case["n_local"] + (own[1] - own[0]) * case["n_src"] * case["n_local"])
    return {"bytes": 2 * moved, "flops": 0}


# ---- 64-bit values --------------------------------------------------------------------------------
def _components(x):
    re = (x >> 4).to(torch.int64)
    im = (x & 15).to(torch.int64)
    return re - 16 * (re > 7), im - 16 * (im > 7)


def _exact_cross(blocks, npol):
    t, c, n = blocks[0].shape
    s = n // npol
    a, b = torch.tril_indices(s, s, device="cuda")
    out = torch.zeros((c, a.numel(), npol, npol, 2), dtype=torch.float64, device="cuda")
    for f in range(c):
        v = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
        for x in blocks:
            re, im = _components(x[:, f])
            z = torch.complex(re.double(), im.double())
            v += z.T @ z.conj()
        v = v.view(s, npol, s, npol).permute(0, 2, 1, 3)[a, b]  # [pairs][p][q]
        out[f] = torch.view_as_real(v)
    return out.view(c, a.numel(), npol * npol, 2)


def _exact_autos(blocks):
    total = 0
    for x in blocks:
        for t0 in range(0, x.shape[0], 64):
            re, im = _components(x[t0:t0 + 64])
            total = total + (re * re + im * im).sum(0)
    return total.double()


def _hamming_sinc(n_taps):
    j = np.arange(n_taps * M, dtype=np.float64)
    last = n_taps * M - 1
    h = (0.54 - 0.46 * np.cos(2.0 * np.pi * j / last)) * np.sinc((j - 0.5 * last) / M)
    return np.floor(h * (131071.0 / np.abs(h).max()) + 0.5)


def exact(case, seed):
    kind = case["kind"]
    if kind == "pfb":
        adc = _pfb_input(case, seed)
        taps, spectra = case["n_taps"], case["n_spectra"]
        h = torch.from_numpy(_hamming_sinc(taps)).cuda().view(taps, M)
        out = torch.empty((case["n_inputs"], spectra, F, 2), dtype=torch.float64, device="cuda")
        for i in range(case["n_inputs"]):
            frames = adc[i].double().view(-1, M)
            y = sum(frames[p:p + spectra] * h[p] for p in range(taps))
            out[i] = torch.view_as_real(torch.fft.rfft(y, dim=1)[:, :F] / M)
        return out
    if case.get("fmt", "ci64") == "ci64" or kind in ("requant", "turn"):
        return None  # whole numbers
    if kind == "autos":
        a = _exact_autos(_blocks(case, seed))
        return {"autos": a / case["n_time"] if case["fmt"] == "cf32_norm" else a}
    shapes = [(case["n_inputs"], case["n_chans"])] if kind == "xengine" else _shapes(case)
    n_time = case["n_time"] * case.get("blocks", 1)
    # 64-bit products at about 1 TFLOP/s, 0.3 ms of launches a channel
    if sum(8.0 * n * n * c * n_time / 1e12 + 3e-4 * c for n, c in shapes) > 15:
        return None
    if kind == "xengine":
        sets = [_blocks(case, seed)]
    else:
        g = _generator(seed)
        sets = [[_samples(g, case["n_time"], c, n)] for n, c in shapes]
    scale = 1.0 / n_time if case["fmt"] == "cf32_norm" else 1.0
    out = []
    for blocks in sets:
        cross, autos = _exact_cross(blocks, case["n_pol"]) * scale, _exact_autos(blocks) * scale
        if case.get("outriggers"):
            st = torch.tensor(_stations(case), device="cuda")
            autos = autos.view(autos.shape[0], -1, case["n_pol"])[:, st]
        out.append({"cross": cross, "autos": autos})
    return out[0] if kind == "xengine" else out
