"""The calls that stand for this framework's use, at sizes from a small
block to the full arrays, for timing and for comparing outputs.

A case is a dict of plain values; ``kind`` names the call:

* ``block``     one context: push a device block, dump its visibilities
                (``Correlator.bind`` / ``push`` / ``dump_into``);
* ``stream``    a dump's blocks in one call, dumps overlapped with the next
                integration (``push_many`` / ``dump_async`` / ``dump_wait``);
* ``pipelined`` blocks that need the corner turn, turned beside the
                cross-multiply (``set_pipeline``), dumps overlapped;
* ``noalloc``   ``corr_correlate_noalloc_bits``, one block, nothing allocated;
* ``batch``     several arrays in one replayed launch (``Batch.run``);
* ``service``   integration requests of several arrays: submit, push, tick,
                fetch (``Service``);
* ``fengine``   ADC samples to packed codes (``FEngine.channelise``);
* ``fx``        ADC samples to visibilities, with the equaliser's power sums;
* ``packets``   a block in packet order to visibilities
                (``PacketRing.turn``, then push and dump);
* ``normalise`` correlation coefficients of an integration
                (``Correlator.normalise_into``).

Sample blocks are quantised Gaussian noise (4-bit: sigma 2.5 clipped to +-7;
8-bit: sigma 20), ADC streams Gaussian noise of sigma 16, as the
configurations of this repository have them; every block is made on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1904_07778_gb300 import xengine as xe
from paper_1904_07778_gb300.fengine import FEngine
from paper_1904_07778_gb300.ingest import PacketRing

TCI, TIC, CIT = xe.CORR_L_TCI, xe.CORR_L_TIC, xe.CORR_L_CIT


def listed():
    return [
        # the smallest calls: a small subarray in a real-time loop that cannot allocate
        {"name": "noalloc_small", "kind": "noalloc", "n": 16, "c": 64, "t": 256, "bits": 4, "layout": TCI},
        # the plain dish array, one 8 MiB block in, its visibilities out: latency
        {"name": "dish_block", "kind": "block", "n": 32, "c": 256, "t": 1024, "bits": 4, "layout": TCI},
        # the dish array's long integration: many packet-order blocks per dump
        {"name": "dish_stream", "kind": "stream", "n": 32, "c": 1024, "t": 4096, "bits": 4, "layout": TCI,
         "blocks": 16},
        # the cylinder array as the receiver groups deliver it: corner turn, then cross-multiply
        {"name": "cylinder_block", "kind": "block", "n": 192, "c": 1024, "t": 8192, "bits": 4, "layout": TIC},
        # the same array streaming, the turn of a block beside the cross-multiply of the one before
        {"name": "cylinder_pipelined", "kind": "pipelined", "n": 192, "c": 1024, "t": 8192, "bits": 4,
         "layout": TIC, "blocks": 3, "turn_sms": 42},
        # an array that fits no tile, vector or swizzle: odd inputs, channels and spectra
        {"name": "ragged_block", "kind": "block", "n": 100, "c": 333, "t": 3001, "bits": 4, "layout": TCI},
        # subarrays of different sizes correlated together
        {"name": "batch_mixed", "kind": "batch", "n": 192, "c": 1024, "t": 8192, "bits": 4, "layout": TCI},
        # the service: 8-bit requests of 512, 192 and 32 inputs, two blocks each
        {"name": "service_mixed", "kind": "service", "n": 512, "c": 256, "t": 4096, "bits": 8, "layout": TCI,
         "blocks": 2},
        # the cylinder array's F-engine: 192 ADC streams to 1024 channels of 4-bit codes
        {"name": "fengine_cylinder", "kind": "fengine", "n": 192, "c": 1024, "t": 2048, "taps": 4, "layout": CIT},
        # the dish array from ADC samples to visibilities, gain statistics on
        {"name": "fx_dish", "kind": "fx", "n": 32, "c": 256, "t": 4096, "taps": 4, "layout": CIT},
        # the network path: F-engine packets as received, turned on the GPU, correlated
        {"name": "packets_cylinder", "kind": "packets", "n": 192, "c": 1024, "t": 1024, "bits": 4, "layout": CIT},
        # monitoring: correlation coefficients of the cylinder's visibilities
        {"name": "normalise_cylinder", "kind": "normalise", "n": 192, "c": 1024, "t": 256, "bits": 4, "layout": TCI},
    ]


_KINDS = ("noalloc", "block", "block", "block", "stream", "pipelined", "batch", "service", "fengine", "fx",
          "packets", "normalise")


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(_KINDS)
    if kind == "noalloc":  # within the fixed scratch
        return {"kind": kind, "n": rng.choice([8, 16, 24, 32, 48, 64]), "c": _log(rng, 8, 128),
                "t": _log(rng, 64, 1024), "bits": 4, "layout": rng.choice([TCI, TIC])}
    if kind == "block":
        bits = rng.choice([4, 4, 8])
        n = rng.choice([_log(rng, 4, 512), rng.choice([16, 32, 64, 96, 128, 192, 256, 384, 512])])
        t = rng.choice([_log(rng, 256, 8192), 1 << rng.randint(8, 13)])
        most = min(1024, (1 << 30) // (n * t * bits // 4), (1 << 30) // (8 * n * (n + 1)))
        return {"kind": kind, "n": n, "c": _log(rng, max(1, most // 16), max(1, most)), "t": t, "bits": bits,
                "layout": rng.choice([TCI, TIC, CIT])}
    if kind == "stream":
        n, t = rng.choice([16, 32, 64, 128]), 16 * _log(rng, 32, 256)
        return {"kind": kind, "n": n, "c": _log(rng, 128, 1024), "t": t, "bits": rng.choice([4, 4, 8]),
                "layout": rng.choice([TCI, CIT]), "blocks": rng.randint(2, 8)}
    if kind == "pipelined":
        return {"kind": kind, "n": rng.choice([96, 128, 192, 256]), "c": 32 * _log(rng, 4, 24),
                "t": 256 * _log(rng, 4, 24), "bits": 4, "layout": TIC, "blocks": rng.randint(2, 3),
                "turn_sms": rng.randint(32, 48)}
    if kind in ("batch", "service"):
        n = rng.choice([64, 128, 192, 256] if kind == "batch" else [192, 256, 384, 512])
        d = {"kind": kind, "n": n, "c": _log(rng, 64, 1024 if kind == "batch" else 256), "t": 16 * _log(rng, 64, 256),
             "bits": 4 if kind == "batch" else 8, "layout": TCI}
        return dict(d, blocks=rng.randint(1, 3)) if kind == "service" else d
    if kind in ("fengine", "fx"):
        c = 1 << rng.randint(6, 11)
        n = rng.choice([_log(rng, 8, 192), rng.choice([32, 64, 192])])
        t = _log(rng, 64, max(64, min(8192, (192 * 1024 * 2048) // (n * c))))
        return {"kind": kind, "n": n, "c": c, "t": t if kind == "fengine" else 16 * (t // 16 + 1),
                "taps": rng.choice([2, 4, 4, 4, 8]), "layout": rng.choice([CIT, CIT, TCI]) if kind == "fengine" else CIT}
    if kind == "packets":
        return {"kind": kind, "n": 32 * rng.randint(1, 6), "c": 32 * _log(rng, 2, 32), "t": 8 * _log(rng, 16, 256),
                "bits": 4, "layout": CIT}
    n = _log(rng, 8, 256)
    return {"kind": kind, "n": n, "c": _log(rng, 16, 1024), "t": 64 * rng.randint(1, 8), "bits": 4, "layout": TCI}


# ------------------------------------------------------------------- inputs
def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + salt)


def _codes(g, count, bits):
    """count packed complex samples (4-bit: one byte each, 8-bit: two), in flat order."""
    out = torch.empty(count * (bits // 4), dtype=torch.uint8, device="cuda")
    step = 1 << 26
    for a in range(0, count, step):
        m = min(step, count - a)
        v = torch.randn(2 * m, generator=g, device="cuda")
        v.mul_(2.5 if bits == 4 else 20.0).round_()
        q = v.clamp_(-7, 7).to(torch.int8) if bits == 4 else v.clamp_(-127, 127).to(torch.int8)
        if bits == 8:
            out[2 * a:2 * (a + m)].copy_(q.view(torch.uint8))
        else:
            u = q.view(torch.uint8)
            torch.bitwise_or(u[:m] << 4, u[m:] & 0xF, out=out[a:a + m])
    return out


def _adc(g, n, samples):
    out = torch.empty((n, samples), dtype=torch.int8, device="cuda")
    for i in range(n):
        v = torch.randn(samples, generator=g, device="cuda").mul_(16.0).round_().clamp_(-127, 127)
        out[i].copy_(v)
    return out


def _gains(case):
    """Equaliser gains (about 10% apart over the band) that bring the codes' RMS near 2.5."""
    c, taps = case["c"], case["taps"]
    m = np.arange(taps * 2 * c, dtype=np.float64)
    size = taps * 2 * c
    h = (0.54 - 0.46 * np.cos(2 * np.pi * m / (size - 1))) * np.sinc((m - (size - 1) / 2) / (2 * c))
    rms = 16.0 * math.sqrt(float((h * h).sum()) / 2)
    band = 1.0 + 0.05 * np.cos(2 * np.pi * np.arange(c) / c)
    g = np.rint(2.5 * 2.0 ** 21 / rms * band)[:, None] * np.ones((1, case["n"]))
    return np.clip(g, 1, (1 << 18) - 1).astype(np.uint32)


def _vis(n, c):
    return torch.zeros((c, n * (n + 1) // 2, 2), dtype=torch.int64, device="cuda")


def _batch_shapes(case):
    """The mixed batch: a small dish array, a mid-size one, and the case's own."""
    return [(32, 256, 1024, 4, TCI), (64, max(1, case["c"] // 2), 4096, 4, TCI),
            (case["n"], case["c"], case["t"], 4, case["layout"])]


def _requests(case):
    """The service's mix: the case's own array, the cylinder and the dish array."""
    t = case["t"]
    return [(case["n"], case["c"], t), (192, 2 * case["c"], t), (32, 4 * case["c"], t)]


def prepare(case, seed):
    kind, n, c, t = case["kind"], case["n"], case["c"], case["t"]
    g = _gen(seed)
    s = {"case": case, "pass": 0}
    if kind == "noalloc":
        s["block"] = _codes(g, n * c * t, case["bits"])
        s["vis"] = _vis(n, c)
        s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind in ("block", "normalise"):
        s["block"] = _codes(g, n * c * t, case["bits"])
        s["cor"] = xe.Correlator(n, c, t, bits=case["bits"], layout=case["layout"])
        if kind == "block":
            s["vis"] = _vis(n, c)
        else:
            s["rho"] = torch.zeros((c, n * (n + 1) // 2, 2), dtype=torch.float64, device="cuda")
            s["cor"].push(s["block"])
            s["cor"].sync()
    elif kind in ("stream", "pipelined"):
        s["blocks"] = [_codes(g, n * c * t, case["bits"]) for _ in range(case["blocks"])]
        s["cor"] = xe.Correlator(n, c, t, bits=case["bits"], layout=case["layout"])
        s["vis"] = [_vis(n, c), _vis(n, c)]
        if kind == "pipelined":
            s["cor"].set_pipeline(case["turn_sms"])
    elif kind == "batch":
        shapes = _batch_shapes(case)
        s["batch"] = xe.Batch(shapes)
        for k, (a, b, d, bits, _) in enumerate(shapes):
            s["batch"].set_input(k, _codes(g, a * b * d, bits))
        s["batch"].sync()
        s["vis"] = [_vis(a, b) for a, b, _, _, _ in shapes]
    elif kind == "service":
        need = 0
        s["blocks"], s["vis"] = [], []
        for a, b, d in _requests(case):
            s["blocks"].append([_codes(g, a * b * d, case["bits"]) for _ in range(case["blocks"])])
            s["vis"].append(_vis(a, b))
            need += a * (a + 1) // 2 * b * 16 + 3 * a * b * d * (case["bits"] // 4) + (1 << 20)
        s["svc"] = xe.Service(need)
    elif kind in ("fengine", "fx"):
        m = 2 * c
        s["adc"] = _adc(g, n, (t + case["taps"] - 1) * m)
        s["fe"] = FEngine(n, c, case["taps"])
        s["fe"].set_gains(_gains(case))
        s["out"] = torch.zeros(n * c * t, dtype=torch.uint8, device="cuda")
        if kind == "fx":
            s["power"] = torch.zeros((c, n), dtype=torch.int64, device="cuda")
            s["cor"] = xe.Correlator(n, c, t, bits=4, layout=CIT)
            s["vis"] = _vis(n, c)
    elif kind == "packets":
        s["ring"] = PacketRing(n // 32, 32, c // 32, 32, t, n_segments=2, packet_order=True)
        s["block"] = _codes(g, n * c * t, 4)
        s["turned"] = torch.zeros(n * c * t, dtype=torch.uint8, device="cuda")
        s["cor"] = xe.Correlator(n, c, t, bits=4, layout=CIT)
        s["vis"] = _vis(n, c)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def _integrate(s, block):
    """Integrate one block in place in the caller's buffer; its dump waits."""
    s["cor"].bind(s["vis"])
    s["cor"].push(block)
    return s["cor"].dump_into(s["vis"])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "noalloc":
        st = xe.corr_correlate_noalloc_bits(s["block"].data_ptr(), case["n"], case["c"], case["t"], case["bits"],
                                            case["layout"], 0, s["vis"].data_ptr(), s["status"].data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        if st != xe.CORR_OK:
            raise xe.CorrError(st, "corr_correlate_noalloc_bits")
        return {"vis": s["vis"], "status": s["status"]}
    if kind == "block":
        return _integrate(s, s["block"])
    if kind in ("stream", "pipelined"):
        # steady state: a dump is waited for once the next one is queued
        vis = s["vis"][s["pass"] & 1]
        s["cor"].bind(vis)
        if kind == "stream":
            s["cor"].push_many(s["blocks"])
        else:
            for b in s["blocks"]:
                s["cor"].push(b)
        s["cor"].dump_async(vis)
        if s["pass"] > 0:
            s["cor"].dump_wait()
        s["pass"] += 1
        return vis
    if kind == "batch":
        # the results leave the batch's buffers, which the next run overwrites
        s["batch"].run()
        for k, v in enumerate(s["vis"]):
            st = xe._lib.corr_batch_get_output(s["batch"]._b, k, v.data_ptr())
            if st != xe.CORR_OK:
                raise xe.CorrError(st, "corr_batch_get_output")
        s["batch"].sync()
        return s["vis"]
    if kind == "service":
        svc = s["svc"]
        ids = [svc.submit(a, b, case["bits"], case["layout"], d, case["blocks"]) for a, b, d in _requests(case)]
        for k in range(case["blocks"]):
            for i, blocks in zip(ids, s["blocks"]):
                svc.push(i, blocks[k])
            svc.tick()
        svc.wait()
        return [svc.fetch(i, v) for i, v in zip(ids, s["vis"])]
    if kind == "fengine":
        s["fe"].channelise(s["adc"], case["t"], out=s["out"], layout=case["layout"])
        return s["out"]
    if kind == "fx":
        s["power"].zero_()
        s["fe"].channelise(s["adc"], case["t"], out=s["out"], layout=case["layout"], power=s["power"])
        return {"vis": _integrate(s, s["out"]), "power": s["power"], "codes": s["out"]}
    if kind == "packets":
        s["ring"].turn(s["block"], s["turned"])
        return _integrate(s, s["turned"])
    return s["cor"].normalise_into(s["rho"])


# -------------------------------------------------------------------- work
def _corr_work(n, c, t, bits):
    nbl = n * (n + 1) // 2
    return {"bytes": n * c * t * (bits // 4) + 16 * nbl * c, "flops": 8 * nbl * c * t}


def _fe_work(case):
    n, c, t, taps = case["n"], case["c"], case["t"], case["taps"]
    m = 2 * c
    return {"bytes": n * (t + taps - 1) * m + n * c * t,
            "flops": n * t * (2 * taps * m + 2.5 * m * math.log2(m))}


def work(case):
    """Bytes read and written once and the operations of one pass: 8 per
    complex multiply-add of the lower triangle; the filter's and half an
    M-point complex transform's per spectrum."""
    kind, n, c, t = case["kind"], case["n"], case["c"], case["t"]
    if kind in ("stream", "pipelined"):
        one = _corr_work(n, c, t * case["blocks"], case["bits"])
    elif kind == "batch":
        parts = [_corr_work(a, b, d, bits) for a, b, d, bits, _ in _batch_shapes(case)]
        one = {k: sum(p[k] for p in parts) for k in parts[0]}
    elif kind == "service":
        parts = [_corr_work(a, b, d * case["blocks"], case["bits"]) for a, b, d in _requests(case)]
        one = {k: sum(p[k] for p in parts) for k in parts[0]}
    elif kind == "fengine":
        one = _fe_work(case)
    elif kind == "fx":
        a, b = _fe_work(case), _corr_work(n, c, t, 4)
        one = {k: a[k] + b[k] for k in a}
    elif kind == "normalise":
        total = n * (n + 1) // 2 * c
        one = {"bytes": 32 * total, "flops": 5 * total}
    else:
        one = _corr_work(n, c, t, case["bits"])
    return {k: float(v) for k, v in one.items()}


def exact(case, seed):
    """The coefficients in 64 bits, straight from the samples; every other
    output is a whole number or a byte."""
    if case["kind"] != "normalise":
        return None
    n, c, t = case["n"], case["c"], case["t"]
    u = _codes(_gen(seed), n * c * t, 4).view(t, c, n).permute(1, 2, 0).to(torch.int16)
    re = (((u >> 4) ^ 8) - 8).double()
    im = (((u & 15) ^ 8) - 8).double()
    i, j = np.tril_indices(n)
    i, j = torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda()
    out = torch.empty((c, i.numel(), 2), dtype=torch.float64, device="cuda")
    for k in range(c):
        r, m = re[k], im[k]
        vr, vi = r @ r.T + m @ m.T, m @ r.T - r @ m.T
        p = vr.diagonal()
        den = torch.sqrt(p[i] * p[j])
        ok = den > 0
        out[k, :, 0] = torch.where(ok, vr[i, j] / torch.where(ok, den, 1.0), 0.0)
        out[k, :, 1] = torch.where(ok, vi[i, j] / torch.where(ok, den, 1.0), 0.0)
    return out
