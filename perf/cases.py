"""The correlator's work as a user has it done, for timing: one pass of each case goes through the
public entry points of the binding (``paper_0910_1517_gb300.corr``) and returns what they compute.

Kinds of case
  fx      one integration from device samples (corr_integrate_device, or corr_integrate_static with
          static=True): visibilities and beams; with dump > 0 the 1 ms auto-power dumps of the RFI
          stage, with block > 0 behind the voltage blanker, with n_beams > 0 phased beams
  push    streaming ingest from pinned host memory (int8, or the 4-bit ADC card rows) with the
          results read from a ring of host slots
  batch   several uneven sub-arrays in one graph launch
  dedisp  one push of a voltage beam through the coherent dedisperser
  flag    power dumps cut into patches, MAD flags, and the learned flagger's probabilities
  grad    the learned flagger's loss and gradients on a batch of patches
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0910_1517_gb300 import corr

SIGMA, RHO = 20.0, 0.05
MODES = {"fp32": corr.CORR_FP32, "i8": corr.CORR_I8, "f16": corr.CORR_F16, "fp32tc": corr.CORR_FP32TC}
TAIL = 2048                      # samples after the last frame: the longest delay
F_LO, BW = 1780.0 / 3.0, 100.0 / 3.0   # MHz: the 610 MHz band
SUBARRAYS = ((8, 2, 512), (16, 2, 1024), (32, 2, 2048), (64, 2, 4096))
NET = ((0, 144, 9), (160, 4608, 144), (4800, 4608, 288), (9424, 16, 16))   # weights: offset, count, fan-in
NET_BIAS = ((144, 16), (4768, 32), (9408, 16))


def _fx(name=None, xmode="fp32", n_ant=32, n_pol=2, n_fft=2048, n_int=8192, beam_avg=1, polself=False, static=False,
        dump=0, block=0, n_beams=0, avg=256):
    c = dict(kind="fx", xmode=xmode, n_ant=n_ant, n_pol=n_pol, n_fft=n_fft, n_int=n_int, beam_avg=beam_avg,
             polself=polself, static=static, dump=dump, block=block, n_beams=n_beams, avg=avg)
    return dict(c, name=name) if name else c


def listed():
    return [
        # four antennas for a fraction of a millisecond: latency and launches
        _fx("fx_tiny", n_ant=4, n_fft=512, n_int=64),
        # an odd antenna count and a ragged integration in the FP16 form
        _fx("fx_odd_f16", "f16", n_ant=11, n_fft=1024, n_int=1040),
        # the 32-antenna dual-polarisation array, 0.25 s, FP32 accuracy on the tensor cores: the main workload
        _fx("fx_gmrt_fp32tc", "fp32tc"),
        # the same array in the default precision mode, two antennas out, averaged beams and power dumps
        _fx("fx_gmrt_fp32", "fp32", n_ant=30, n_int=4096, beam_avg=8, dump=32),
        # the int8 precision form of the main workload
        _fx("fx_gmrt_i8", "i8"),
        # RFI-hit samples behind the voltage blanker
        _fx("fx_gmrt_blank", "fp32tc", n_int=4096, block=16384),
        # 16 phased beams with full-polar products beside the correlation
        _fx("fx_gmrt_beams16", "fp32tc", n_int=4096, n_beams=16),
        # four concurrent observations of uneven sizes, 8 to 64 antennas and 512- to 4096-point FFTs
        dict(name="batch4_i8", kind="batch", xmode="i8", n_sub=4, first=0, n_int=4096),
        # live 4-bit ADC data arriving from the host, results back to the host
        dict(name="push_4bit", kind="push", bits=4, xmode="fp32tc", n_ant=32, n_pol=2, n_fft=2048, n_int=1024),
        # a millisecond pulsar's voltage beam: 33 MHz at 610 MHz, DM 30
        dict(name="dedisp_610", kind="dedisp", n_chan=1024, frames=4096, overlap=1200, push=8192, avg=64, dm=30.0),
        # flagging one integration's power dumps: 4096 patches
        dict(name="flag_4096", kind="flag", n_in=64, n_dump=256, n_chan=1024),
        # one training batch
        dict(name="grad_256", kind="grad", batch=256),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _array(rng, most):
    """n_ant, n_pol, n_fft, n_int with at most `most` samples in all."""
    n_pol = rng.choice((1, 2, 2))
    n_ant = max(2, min(128 // n_pol, round(_log(rng, 2, 64))))
    n_fft = 1 << rng.randint(6, 12)
    top = max(16, min(8192, most // (n_ant * n_pol * n_fft)))
    n_int = max(16, round(_log(rng, 16, top)) // 16 * 16)
    return n_ant, n_pol, n_fft, n_int


def draw(rng):
    kind = rng.choice(("fx",) * 7 + ("push", "batch", "dedisp", "flag", "grad"))
    if kind == "fx":
        n_ant, n_pol, n_fft, n_int = _array(rng, 1 << 29)
        more = rng.choice(("", "", "avg", "dump", "block", "beams"))
        xmode = rng.choice(tuple(MODES))
        if more in ("dump", "beams"):
            xmode = rng.choice(("fp32", "fp32tc"))
        n_beams = 0
        if more == "beams":
            n_beams = round(_log(rng, 1, 64))
            n_int = max(64, min(n_int, (1 << 27) // (n_beams * n_fft)) // 64 * 64)
        spec = n_fft // 2 * n_int * 8 * (n_ant * n_pol + 3)
        static = not more and xmode == "fp32" and n_ant <= 64 and spec < (24 << 20)
        return _fx(None, xmode, n_ant, n_pol, n_fft, n_int, beam_avg=rng.choice((2, 8, 16)) if more == "avg" else 1,
                   polself=not static and rng.random() < 0.2, static=static, dump=16 if more == "dump" else 0,
                   block=rng.choice((4096, 8192, 16384, 32768)) if more == "block" else 0, n_beams=n_beams,
                   avg=rng.choice((1, 8, 64)) if n_beams * n_int * n_fft < 1 << 23 else 64)
    if kind == "push":
        n_ant, n_pol, n_fft, n_int = _array(rng, 1 << 27)
        bits = rng.choice((4, 8))
        if bits == 4:
            n_ant = max(4, n_ant // 4 * 4)
        return dict(kind="push", bits=bits, xmode=rng.choice(("fp32", "fp32tc", "i8")), n_ant=n_ant, n_pol=n_pol,
                    n_fft=n_fft, n_int=n_int)
    if kind == "batch":
        n_sub = rng.randint(1, 4)
        return dict(kind="batch", xmode=rng.choice(("fp32", "i8", "f16")), n_sub=n_sub, first=rng.randint(0, 4 - n_sub),
                    n_int=round(_log(rng, 64, 2048)) // 16 * 16)
    if kind == "dedisp":
        n_chan = 1 << rng.randint(6, 12)
        frames = min(1 << rng.randint(8, 12), (1 << 22) // n_chan)
        overlap = rng.randint(frames // 8, frames // 2)
        avg = 1 << rng.randint(1, int(math.log2(n_chan)))
        dm = 0.95 * overlap * n_chan / (4.148808e9 * BW * (F_LO ** -2 - (F_LO + BW) ** -2))
        return dict(kind="dedisp", n_chan=n_chan, frames=frames, overlap=overlap, avg=avg, dm=dm,
                    push=max(frames, min((1 << 23) // n_chan, rng.randint(frames, 4 * frames))))
    if kind == "flag":
        return dict(kind="flag", n_in=rng.randint(1, 64), n_dump=64 * rng.randint(1, 4), n_chan=64 * rng.randint(1, 16))
    return dict(kind="grad", batch=max(1, round(_log(rng, 1, 256))))


# ---------------------------------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _model(seed, n_ant):
    """Per-antenna delays (samples), fringe phases (rad) and rates (rad per frame), beam weights."""
    r = np.random.default_rng([int(seed), 7])
    delay = r.uniform(0, 2000.0, n_ant)
    phi0, rate = r.uniform(-math.pi, math.pi, n_ant), r.uniform(0, 0.1, n_ant)
    coh = np.ones(n_ant, np.uint8)
    coh[max(1, n_ant - 2):] = 0
    return delay, phi0, rate, coh


def _samples(seed, n_ant, n_pol, n, delay, bursts=False):
    """int8 [n_in][ld]: Gaussian receiver noise, a common sky signal that reaches antenna a delay[a]
    samples late, optionally broadband bursts over 2.5 % of the time."""
    g = _gen(seed)
    D = np.floor(np.asarray(delay) + 0.5).astype(int)
    ld = (n + 15) // 16 * 16 + 16
    x = torch.zeros((n_ant * n_pol, ld), dtype=torch.int8, device="cuda")
    idx = None
    if bursts:
        start = torch.randint(0, n - 100, (max(1, n // 4000),), generator=g, device="cuda")
        idx = (start[:, None] + torch.arange(100, device="cuda")[None, :]).reshape(-1)
    for p in range(n_pol):
        sky = torch.randn(n + 2048, generator=g, device="cuda")
        for a in range(n_ant):
            v = torch.randn(n, generator=g, device="cuda").mul_(math.sqrt(1 - RHO) * SIGMA)
            v.add_(sky[2048 - D[a]:2048 - D[a] + n], alpha=math.sqrt(RHO) * SIGMA)
            if idx is not None:
                v[idx] += 90.0 * (1 if (a + p) % 2 else -1)
            x[a * n_pol + p, :n] = v.round_().clamp_(-127, 127).to(torch.int8)
    return x


def _scales(n_in, n_chan):
    """Requantisation scales 127 / (4 sigma) of the nominal input level; at DC one component has all the power."""
    s = np.full((n_in, n_chan), 127.0 / (4.0 * SIGMA * math.sqrt(n_chan)), np.float32)
    s[:, 0] = 127.0 / (4.0 * SIGMA * math.sqrt(2.0 * n_chan))
    return s


def _beam_weights(seed, n_beams, n_ant, n_chan):
    r = np.random.default_rng([int(seed), 9])
    return np.exp(2j * np.pi * r.uniform(-20, 20, (n_beams, n_ant, 1)) * np.arange(n_chan)[None, None, :] /
                  (2 * n_chan)).astype(np.complex64)


def _noise(seed, n_in):
    return np.random.default_rng([int(seed), 11]).standard_normal((n_in, 1 << 16)).astype(np.float32)


def _net_params(seed):
    r = np.random.default_rng([int(seed), 13])
    p = np.zeros(9441, np.float32)
    for o, n, fan in NET:
        p[o:o + n] = r.normal(scale=math.sqrt(2.0 / fan), size=n)
    for o, n in NET_BIAS:
        p[o:o + n] = 0.05
    return p


def _dumps(seed, n_in, n_dump, n_chan):
    """Power dumps of 32 frames (sums of 32 exponential variates) with tones and broadband bursts, and the mask."""
    g = _gen(seed)
    P = torch.zeros((n_in, n_dump, n_chan), device="cuda")
    for _ in range(32):
        P -= torch.log(torch.rand(P.shape, generator=g, device="cuda").clamp_min_(1e-7))
    mask = torch.zeros(P.shape, dtype=torch.uint8, device="cuda")
    tone = torch.rand((n_in, 1, n_chan), generator=g, device="cuda") < 0.03
    on = (torch.arange(n_dump, device="cuda")[None, :, None] // 16 + torch.arange(n_chan, device="cuda")) % 3 > 0
    burst = torch.rand((n_in, n_dump, 1), generator=g, device="cuda") < 0.01
    mask |= ((tone & on) | burst).to(torch.uint8)
    kappa = 5.0 * torch.exp(2.3 * torch.rand((n_in, n_dump, n_chan), generator=g, device="cuda"))
    P += mask * kappa * math.sqrt(32.0)
    return (P * (2 * n_chan * SIGMA ** 2)).contiguous(), mask


def _cut(P):
    """[n_in][n_dump][n_chan] into 64 x 64 patches."""
    a, d, k = P.shape
    return P.reshape(a, d // 64, 64, k // 64, 64).permute(0, 1, 3, 2, 4).reshape(-1, 64, 64).contiguous()


def _patch_input(P):
    """The network input of power dumps in 64 bits: sign(u) log(1 + |u|), and median, MAD and deviations."""
    v = _cut(P).double().reshape(-1, 4096)

    def mid(t):
        s = t.sort(dim=1).values
        return 0.5 * (s[:, 2047] + s[:, 2048])
    med = mid(v)
    dev = v - med[:, None]
    mad = mid(dev.abs())
    u = dev / (mad / 0.6745)[:, None]
    return torch.sign(u) * torch.log1p(u.abs()), med, mad, dev


class _Owner(list):
    """The library's objects of one state, as (destroy, object): destroyed when neither the state nor a view of
    their memory is left."""

    def __del__(self):
        for f, v in self:
            f(v)


class _Array:
    """float32 device memory of the library, as torch takes it; the tensor keeps the owner alive."""

    def __init__(self, owner, ptr, shape):
        self.owner = owner
        self.__cuda_array_interface__ = dict(shape=tuple(shape), typestr="<f4", data=(int(ptr), False), version=2)


def _view(owner, ptr, shape):
    return torch.as_tensor(_Array(owner, ptr, shape), device="cuda")


# --------------------------------------------------------------------------------------- prepare


def _handle(own, seed, n_ant, n_pol, n_fft, n_int, xmode, polself=False, beam_avg=1):
    delay, phi0, rate, coh = _model(seed, n_ant)
    h = corr.corr_create(n_ant, n_pol, n_fft, n_int)
    own.append((corr.corr_destroy, h))
    corr.corr_set_delays(h, delay, phi0, rate)
    corr.corr_set_beam_weights(h, None, None, None, coh)
    if xmode in ("i8", "f16"):
        corr.corr_set_scales(h, _scales(n_ant * n_pol, n_fft // 2))
    corr.corr_set_mode(h, MODES[xmode], 1 if polself else 0, beam_avg)
    return h


def _outputs(own, h, n_ant, n_pol, n_fft, n_int, polself=False, beam_avg=1):
    vis, beams, _ = corr.corr_device_outputs(h)
    npp = n_pol if polself else n_pol * n_pol
    return (_view(own, vis, (n_fft // 2, n_ant * (n_ant + 1) // 2, npp, 2)),
            _view(own, beams, (2, n_int // beam_avg, n_fft // 2)))


def prepare(case, seed):
    c, own = case, _Owner()
    st, kind = dict(case=case, own=own), case["kind"]
    if kind == "fx":
        size = c["n_ant"], c["n_pol"], c["n_fft"], c["n_int"]
        delay, phi0, rate, _ = _model(seed, c["n_ant"])
        n = c["n_int"] * c["n_fft"] + TAIL
        st["x"], st["n"] = _samples(seed, c["n_ant"], c["n_pol"], n, delay, c["block"] > 0), n
        if c["static"]:
            st["model"] = delay, phi0, rate
            st["vis"] = torch.empty((c["n_fft"] // 2, c["n_ant"] * (c["n_ant"] + 1) // 2, c["n_pol"] ** 2, 2), device="cuda")
            st["beams"] = torch.empty((2, c["n_int"], c["n_fft"] // 2), device="cuda")
            return st
        h = st["h"] = _handle(own, seed, *size, c["xmode"], c["polself"], c["beam_avg"])
        n_in, n_chan = c["n_ant"] * c["n_pol"], c["n_fft"] // 2
        if c["block"]:
            corr.corr_set_blanker(h, 3.0, c["block"], _noise(seed, n_in))
        if c["n_beams"]:
            corr.corr_set_multibeam(h, _beam_weights(seed, c["n_beams"], c["n_ant"], n_chan), 0, c["avg"])
        st["out"] = list(_outputs(own, h, *size, c["polself"], c["beam_avg"]))
        if c["dump"]:
            corr.corr_set_power_dump(h, c["dump"])
            st["out"].append(_view(own, corr.corr_power_device(h), (n_in, c["n_int"] // c["dump"], n_chan)))
    elif kind == "push":
        size = c["n_ant"], c["n_pol"], c["n_fft"], c["n_int"]
        delay, body = _model(seed, c["n_ant"])[0], c["n_int"] * c["n_fft"]
        x = _push_samples(c, seed, delay)
        h = st["h"] = _handle(own, seed, *size, c["xmode"])
        host = _pack(x) if c["bits"] == 4 else x
        per = 2 if c["bits"] == 4 else 1                       # bytes a sample of one row
        cut = (body + TAIL) * per
        first, st["x"] = (host[:, a:b].contiguous().cpu().pin_memory() for a, b in ((0, cut), (cut, cut + body * per)))
        st["vis"] = torch.empty((2, c["n_fft"] // 2, c["n_ant"] * (c["n_ant"] + 1) // 2, c["n_pol"] ** 2, 2)).pin_memory()
        st["beams"] = torch.empty((2, 2, c["n_int"], c["n_fft"] // 2)).pin_memory()
        corr.corr_set_output_ring(h, st["vis"], st["beams"], 2)
        st["seq"] = _push(st, first, body + TAIL, 0)
        corr.corr_wait_output(h, 0)
        st["index"] = 1
    elif kind == "batch":
        st["hs"], st["xs"], st["out"] = [], [], []
        for q in range(c["first"], c["first"] + c["n_sub"]):
            n_ant, n_pol, n_fft = SUBARRAYS[q]
            h = _handle(own, seed + q, n_ant, n_pol, n_fft, c["n_int"], c["xmode"])
            n = c["n_int"] * n_fft + TAIL
            st["hs"].append(h)
            st["xs"].append(_samples(seed + q, n_ant, n_pol, n, _model(seed + q, n_ant)[0]))
            st["out"].append(_outputs(own, h, n_ant, n_pol, n_fft, c["n_int"]))
        st["b"] = corr.corr_batch_create(st["hs"])
        own.insert(0, (corr.corr_batch_destroy, st["b"]))
        st["n"] = [x.shape[1] for x in st["xs"]]
    elif kind == "dedisp":
        d = st["d"] = corr.corr_dd_create(c["n_chan"], c["frames"], c["overlap"], c["push"], c["dm"], F_LO, BW,
                                          c["avg"])
        own.append((corr.corr_dd_destroy, d))
        st["x"] = torch.randn((c["push"], c["n_chan"], 4), generator=_gen(seed), device="cuda") * 100.0
        keep = c["frames"] - c["overlap"]
        st["y"] = torch.zeros((c["push"] // keep + 1) * keep * c["n_chan"] // c["avg"], device="cuda")
    else:
        n_in, n_dump, n_chan = (c["n_in"], c["n_dump"], c["n_chan"]) if kind == "flag" else (c["batch"], 64, 64)
        P, mask = _dumps(seed, n_in, n_dump, n_chan)
        B = n_in * (n_dump // 64) * (n_chan // 64)
        net = st["net"] = corr.rfi_create(min(B, 1024))
        own.append((corr.rfi_destroy, net))
        corr.rfi_set_params(net, _net_params(seed))
        st["x"] = torch.empty((B, 64, 64), dtype=torch.float16, device="cuda")
        if kind == "flag":
            st["P"], st["flags"] = P, torch.empty((B, 64, 64), dtype=torch.uint8, device="cuda")
            st["stats"], st["prob"] = torch.empty((B, 2), device="cuda"), torch.empty((B, 64, 64), device="cuda")
        else:
            st["x"].copy_(_patch_input(P)[0].reshape(B, 64, 64))
            st["mask"] = _cut(mask)
    return st


def _push_samples(c, seed, delay):
    x = _samples(seed, c["n_ant"], c["n_pol"], 2 * c["n_int"] * c["n_fft"] + TAIL, delay)
    return (x.float() / 5.0).round_().clamp_(-8, 7).to(torch.int8) if c["bits"] == 4 else x


def _pack(x):
    """ADC card rows: 4 inputs x 4 bits in two bytes a sample."""
    n = (x.to(torch.uint8) & 15).reshape(x.shape[0] // 4, 4, x.shape[1])
    return torch.stack((n[:, 0] | (n[:, 1] << 4), n[:, 2] | (n[:, 3] << 4)), dim=2).reshape(n.shape[0], -1)


def _push(st, x, n, seq):
    if st["case"]["bits"] == 4:
        corr.corr_push_samples_4bit(st["h"], x, n, seq)
    else:
        corr.corr_push_samples(st["h"], x, seq)
    return seq + n


# ------------------------------------------------------------------------------------------- run


def run(state):
    st, c = state, state["case"]
    kind, stream = c["kind"], torch.cuda.current_stream()
    if kind == "fx":
        if c["static"]:
            delay, phi0, rate = st["model"]
            corr.corr_integrate_static(c["n_ant"], c["n_pol"], c["n_fft"], c["n_int"], st["x"], st["vis"], st["beams"],
                                       delay, phi0, rate, n_avail=st["n"], stream=stream, blocking=0)
            return [st["vis"], st["beams"]]
        corr.corr_integrate_device(st["h"], st["x"], n_avail=st["n"], stream=stream)
        if c["n_beams"]:                                       # read by copy: they have no device pointer
            return st["out"] + [corr.corr_read_multibeam(st["h"], c["n_beams"], c["n_int"] // c["avg"])]
        return st["out"]
    if kind == "push":
        j = st["index"]
        st["seq"] = _push(st, st["x"], c["n_int"] * c["n_fft"], st["seq"])
        slot = corr.corr_wait_output(st["h"], j)
        st["index"] = j + 1
        return [st["vis"][slot], st["beams"][slot]]
    if kind == "batch":
        corr.corr_batch_integrate_device(st["b"], st["xs"], n_avail=st["n"], stream=stream)
        return st["out"]
    if kind == "dedisp":
        n = corr.corr_dd_push_device(st["d"], st["x"], st["y"], stream=stream)
        return st["y"][:n]
    if kind == "flag":
        corr.rfi_patches(st["P"], c["n_in"], c["n_dump"], c["n_chan"], 5.0, st["x"], st["flags"], st["stats"], stream=stream)
        for b in range(0, st["x"].shape[0], 1024):
            part = st["x"][b:b + 1024]
            corr.rfi_infer(st["net"], part, part.shape[0], st["prob"][b:b + 1024], stream=stream)
        return [st["x"], st["flags"], st["stats"], st["prob"]]
    loss, grad = corr.rfi_loss_grad(st["net"], st["x"], st["mask"], c["batch"], stream=stream)
    return [loss, grad]


# ------------------------------------------------------------------------------------------ work


def _fx_work(n_ant, n_pol, n_fft, n_int, polself=False, beam_avg=1):
    n_in, n_chan = n_ant * n_pol, n_fft // 2
    s = n_in * n_int * n_fft
    npp = n_pol if polself else n_pol * n_pol
    b = s + n_chan * n_ant * (n_ant + 1) // 2 * npp * 8 + 2 * n_int // beam_avg * n_chan * 4
    macs = n_ant * (n_ant + 1) / 2 * npp
    return b, s * (2.5 * math.log2(n_fft) + 9) + 8.0 * macs * n_chan * n_int


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        w = [_fx_work(*SUBARRAYS[q], c["n_int"]) for q in range(c["first"], c["first"] + c["n_sub"])]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    if kind in ("fx", "push"):
        b, f = _fx_work(c["n_ant"], c["n_pol"], c["n_fft"], c["n_int"], c.get("polself", False), c.get("beam_avg", 1))
        s = c["n_ant"] * c["n_pol"] * c["n_int"] * c["n_fft"]
        if kind == "push":
            return {"bytes": b - (s // 2 if c["bits"] == 4 else 0), "flops": f}
        if c["dump"]:
            b, f = b + s // 2 // c["dump"] * 4, f + 2 * s
        if c["n_beams"]:
            b, f = b + c["n_beams"] * (c["n_int"] // c["avg"]) * c["n_fft"] // 2 * 16, f + 4.0 * c["n_beams"] * s
        return {"bytes": b, "flops": f}
    if kind == "dedisp":
        n, M = c["push"] * c["n_chan"], c["frames"] * c["n_chan"]
        over = c["frames"] / (c["frames"] - c["overlap"])
        return {"bytes": 16 * n + 4 * n // c["avg"],
                "flops": 2 * n * (5 * math.log2(c["n_chan"]) + over * (10 * math.log2(M) + 6) + 3)}
    if kind == "flag":
        px = c["n_in"] * c["n_dump"] * c["n_chan"]
        return {"bytes": px * (4 + 2 + 1 + 4), "flops": px * 2.0 * 9376}
    return {"bytes": c["batch"] * 4096 * 3 + 9441 * 4, "flops": c["batch"] * 4096 * 2.0 * (3 * 9376 - 144)}


# ----------------------------------------------------------------------------------------- exact


def _spectra(x, c, model, g0, t0, t1):
    """Y [n_in][t1 - t0][n_chan] complex128 of frames t0 .. t1 - 1."""
    n_ant, n_pol, N = c["n_ant"], c["n_pol"], c["n_fft"]
    delay, phi0, rate, _ = model
    Y = torch.empty((n_ant * n_pol, t1 - t0, N // 2), dtype=torch.complex128, device="cuda")
    k = torch.arange(N // 2, dtype=torch.float64, device="cuda")
    t = torch.arange(t0, t1, dtype=torch.float64, device="cuda") + g0
    for a in range(n_ant):
        D = math.floor(delay[a] + 0.5)
        fr = -(phi0[a] + rate[a] * t)
        ph = 2 * math.pi * (delay[a] - D) / N * k
        w = torch.polar(torch.ones_like(ph), ph)[None, :] * torch.polar(torch.ones_like(fr), fr)[:, None]
        for p in range(n_pol):
            row = x[a * n_pol + p, D + t0 * N:D + t1 * N].double().reshape(t1 - t0, N)
            Y[a * n_pol + p] = torch.fft.rfft(row)[:, :N // 2] * w
    return Y


def _exact_fx(x, c, model, g0=0, scales=None, dump=0, weights=None, avg=1):
    """Visibilities, beams, power dumps and phased beams in 64 bits, a block of frames at a time."""
    n_ant, n_pol, n_chan, n_int = c["n_ant"], c["n_pol"], c["n_fft"] // 2, c["n_int"]
    n_in, coh = n_ant * n_pol, model[3]
    per = max(256, 1 << max(4, int(math.log2(2e8 / (n_in * n_chan)))))    # a multiple of every window
    G = torch.zeros((n_chan, n_in, n_in), dtype=torch.complex128, device="cuda")
    inc, cohb, dumps, mb = [], [], [], []
    w = None if weights is None else torch.from_numpy(weights).cuda().to(torch.complex128).permute(2, 0, 1)
    s = None if scales is None else torch.from_numpy(scales).cuda().double()
    for t0 in range(0, n_int, per):
        Y = _spectra(x, c, model, g0, t0, min(n_int, t0 + per))
        n = Y.shape[1]
        P = Y.real.square() + Y.imag.square()
        inc.append(P.sum(0))
        B = sum(Y[[i for i in range(n_in) if i % n_pol == p and coh[i // n_pol]]].sum(0).abs().square() for p in range(n_pol))
        cohb.append(B)
        if dump:
            dumps.append(P.reshape(n_in, n // dump, dump, n_chan).sum(2))
        del P
        Yk = Y.permute(2, 0, 1).contiguous()                              # [k][input][frame]
        del Y
        if w is not None:
            U = [torch.matmul(w, Yk[:, p::n_pol]) for p in range(n_pol)]  # [k][beam][frame]
            z = torch.zeros_like(U[0].real)
            X = U[0] * U[1].conj() if n_pol == 2 else None
            o = [U[0].abs().square(), U[1].abs().square() if n_pol == 2 else z, X.real if n_pol == 2 else z,
                 X.imag if n_pol == 2 else z]
            mb.append(torch.stack([v.reshape(n_chan, -1, n // avg, avg).mean(3) for v in o], -1).permute(1, 2, 0, 3))
        if s is not None:
            sk = s.t()[:, :, None]
            Yk.mul_(sk)
            if c["xmode"] == "i8":
                Yk = torch.complex(Yk.real.round().clamp_(-127, 127), Yk.imag.round().clamp_(-127, 127))
            Yk.div_(sk)
        for k in range(0, n_chan, 256):
            G[k:k + 256] += torch.matmul(Yk[k:k + 256], Yk[k:k + 256].mH)
        del Yk
    a, b = np.triu_indices(n_ant)
    prods = [(p, p) for p in range(n_pol)] if c.get("polself") else [(p, q) for p in range(n_pol) for q in range(n_pol)]
    ia = torch.tensor([[i * n_pol + p for p, _ in prods] for i in a], device="cuda")
    ib = torch.tensor([[i * n_pol + q for _, q in prods] for i in b], device="cuda")
    vis = torch.view_as_real(G[:, ia, ib].contiguous())
    beams = torch.stack((torch.cat(inc), torch.cat(cohb)))
    m = c.get("beam_avg", 1)
    out = [vis, beams.reshape(2, n_int // m, m, n_chan).mean(2)]
    return out + ([torch.cat(dumps, 1)] if dump else []) + ([torch.cat(mb, 1)] if mb else [])


def _blanked(x, c, seed, n):
    """The voltage blanker (median / MAD per block of each row, M = 3) on int8 rows."""
    block, noise = c["block"], torch.from_numpy(_noise(seed, x.shape[0])).cuda()
    y = x.clone()
    for i in range(x.shape[0]):
        for p0 in range(0, n, block):
            v = x[i, p0:min(n, p0 + block)].double()

            def mid(t):
                s = t.sort().values
                return 0.5 * (s[(len(s) - 1) // 2] + s[len(s) // 2])
            dev = (v - mid(v)).abs()
            mad = mid(dev)
            g = noise[i, torch.arange(p0, p0 + len(v), device="cuda") % noise.shape[1]]
            r = ((mad / 0.6745).float() * g).round().clamp_(-127, 127).to(torch.int8)
            y[i, p0:p0 + len(v)] = torch.where(dev > 3.0 * mad / 0.6745, r, x[i, p0:p0 + len(v)])
    return y


def _exact_net(c, seed, z, mask=None):
    p = torch.from_numpy(_net_params(seed)).cuda().double().requires_grad_(mask is not None)
    F = torch.nn.functional

    def logits(v):
        a = F.relu(F.conv2d(v, p[0:144].view(16, 1, 3, 3), p[144:160], padding=1))
        a = F.relu(F.conv2d(a, p[160:4768].view(32, 16, 3, 3), p[4768:4800], padding=1))
        a = F.relu(F.conv2d(a, p[4800:9408].view(16, 32, 3, 3), p[9408:9424], padding=1))
        return F.conv2d(a, p[9424:9440].view(1, 16, 1, 1), p[9440:9441])[:, 0]
    z = z.reshape(-1, 1, 64, 64)
    if mask is None:
        with torch.no_grad():
            return torch.cat([torch.sigmoid(logits(v)) for v in z.split(128)])
    loss = 0.0
    for v, m in zip(z.split(64), mask.split(64)):
        part = F.binary_cross_entropy_with_logits(logits(v), m.double(), reduction="sum") / z.numel()
        part.backward()
        loss += float(part)
    return [loss, p.grad.detach().cpu().numpy()]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "fx":
        model, n_in, n_chan = _model(seed, c["n_ant"]), c["n_ant"] * c["n_pol"], c["n_fft"] // 2
        n = c["n_int"] * c["n_fft"] + TAIL
        x = _samples(seed, c["n_ant"], c["n_pol"], n, model[0], c["block"] > 0)
        if c["static"]:
            model = (*model[:3], np.ones(c["n_ant"], np.uint8))
        if c["block"]:
            n = c["n_int"] * c["n_fft"] + int(np.floor(model[0] + 0.5).max())
            if n_in * n // c["block"] > 70000:                 # blocks taken one by one
                return None
            x = _blanked(x, c, seed, n)
        w = _beam_weights(seed, c["n_beams"], c["n_ant"], n_chan) if c["n_beams"] else None
        s = _scales(n_in, n_chan) if c["xmode"] == "i8" else None
        return _exact_fx(x, c, model, scales=s, dump=c["dump"], weights=w, avg=c["avg"])
    if kind == "push":
        model, body = _model(seed, c["n_ant"]), c["n_int"] * c["n_fft"]
        x = _push_samples(c, seed, model[0])
        s = _scales(c["n_ant"] * c["n_pol"], c["n_fft"] // 2) if c["xmode"] == "i8" else None
        return _exact_fx(x[:, body:], c, model, g0=c["n_int"], scales=s)
    if kind == "batch":
        out = []
        for q in range(c["first"], c["first"] + c["n_sub"]):
            n_ant, n_pol, n_fft = SUBARRAYS[q]
            model = _model(seed + q, n_ant)
            x = _samples(seed + q, n_ant, n_pol, c["n_int"] * n_fft + TAIL, model[0])
            s = _scales(n_ant * n_pol, n_fft // 2) if c["xmode"] == "i8" else None
            out.append(_exact_fx(x, dict(n_ant=n_ant, n_pol=n_pol, n_fft=n_fft, n_int=c["n_int"], xmode=c["xmode"]),
                                 model, scales=s))
        return out
    if kind == "dedisp":
        spec = (torch.randn((c["push"], c["n_chan"], 4), generator=_gen(seed), device="cuda") * 100.0).double()
        z = torch.fft.ifft(torch.view_as_complex(spec.reshape(c["push"], c["n_chan"], 2, 2)), dim=1).reshape(-1, 2)
        del spec
        M, keep = c["frames"] * c["n_chan"], c["frames"] - c["overlap"]
        nu = F_LO + torch.arange(M, dtype=torch.float64, device="cuda") * (BW / M)
        ref = F_LO + BW
        cyc = 1e6 * 4.148808e3 * c["dm"] * (nu - ref) ** 2 / (ref * ref * nu)
        ph = -2 * math.pi * (cyc - cyc.floor())
        C = torch.polar(torch.ones_like(ph), ph)[:, None]
        out = []
        for b in range((c["push"] - c["frames"]) // keep + 1):
            y = torch.fft.ifft(torch.fft.fft(z[b * keep * c["n_chan"]:b * keep * c["n_chan"] + M], dim=0) * C, dim=0)
            out.append(y[:keep * c["n_chan"]].abs().square().sum(1).reshape(-1, c["avg"]).mean(1))
        return torch.cat(out)
    n_in, n_dump, n_chan = (c["n_in"], c["n_dump"], c["n_chan"]) if kind == "flag" else (c["batch"], 64, 64)
    P, mask = _dumps(seed, n_in, n_dump, n_chan)
    z, med, mad, dev = _patch_input(P)
    if kind == "grad":
        return _exact_net(c, seed, z.half().double(), _cut(mask))
    flags = (dev.abs() > 5.0 * (mad / 0.6745)[:, None]).to(torch.uint8).reshape(-1, 64, 64)
    return [z.reshape(-1, 64, 64), flags, torch.stack((med, mad), 1), _exact_net(c, seed, z)]
