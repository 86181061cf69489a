"""The decoder's performance cases: what programs that use this library call.

One reconciliation session is Bob's side (his message M and the syndrome),
Alice's LLR map, and the decode; a service runs many sessions at once. The
cases take each of these through the public entry points
(``paper_1702_07740_gb300.qcldpc``), from one short frame to the sixteen
n = 10^6 frames of the benchmark, over the schedules, message formats, maps
and code families the library offers.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU, the code handles and buffers
    run(state)           one pass; returns its outputs
    work(case)           bytes and operations of one pass
    exact(case, seed)    the outputs in 64-bit arithmetic, where they have one

Inputs are synthetic channel draws (x ~ N(0, 1), y = x + N(0, 1/snr), uniform
bits) made with torch's seeded generator; Bob's syndrome, his message and the
LLRs given to the decode cases are formed here in plain torch.
"""
from __future__ import annotations

import functools
import math

import torch

import synth
from paper_1702_07740_gb300 import qcldpc as q

CODES = {"r002": synth.rate002_code, "r005": synth.rate005_code, "r010": synth.rate010_code,
         "met": synth.met_code}
# (base rows, base columns, heavy circulants, degree-1 circulants)
BASE = {"r002": (49, 50, 119, 48), "r005": (19, 20, 38, 19), "r010": (9, 10, 18, 9),
        "met": (1568, 1600, 3812, 1536)}
FMT = {"fp32": 0, "fp16": 1, "int8": 2}
# Three rates, each at three lengths: the mixed workload of the batching study.
MIX = (("r002", 2000), ("r002", 8000), ("r002", 20000), ("r005", 5000), ("r005", 20000),
       ("r005", 50000), ("r010", 10000), ("r010", 40000), ("r010", 100000))
MIX_SNR = {"r002": 0.16, "r005": 0.5, "r010": 1.0}


def listed() -> list:
    return [
        # The smallest session: Bob's message and syndrome and Alice's LLRs of
        # one n = 25,600 frame. Launches and call overhead are all of it.
        dict(name="maps_short", kind="maps", code="r002", Z=512, frames=1, snr=0.029, d=8),
        # The same for a batch of sixteen n = 10^6 frames (130 MB in and out).
        dict(name="maps_batch", kind="maps", code="r002", Z=20000, frames=16, snr=0.029, d=8),
        # The two-dimensional map, which a session may choose instead.
        dict(name="maps_d2", kind="maps", code="r005", Z=50000, frames=4, snr=0.5, d=2),
        # One short frame, posteriors wanted, 50 fixed iterations: the parity
        # workload, and what a low-latency link decodes.
        dict(name="soft_short", kind="decode", code="r002", Z=512, frames=1, snr=0.029, max_iter=50,
             et_start=51, fmt="fp32", soft=True, layers=-1, iters=50),
        # One n = 10^6 frame alone: latency, the GPU partly filled.
        dict(name="one_frame", kind="decode", code="r002", Z=20000, frames=1, snr=0.029, max_iter=100,
             et_start=1, fmt="fp32", soft=False, layers=-1, iters=100),
        # The benchmark: sixteen n = 10^6 frames at the paper's SNR, LLR map
        # and up to 500 iterations with the stop test after each.
        dict(name="paper", kind="alice", code="r002", Z=20000, frames=16, snr=0.029, max_iter=500,
             et_start=1, fmt="fp32", soft=False, layers=-1, iters=500),
        # The same code where frames converge after a few iterations, so the
        # set-up and output steps weigh as much as the loop.
        dict(name="converging", kind="decode", code="r002", Z=20000, frames=16, snr=0.16, max_iter=500,
             et_start=1, fmt="fp32", soft=False, layers=-1, iters=6),
        # Odd lifting size, a ragged handful of frames, int8 messages.
        dict(name="int8_odd", kind="decode", code="r010", Z=9999, frames=7, snr=1.0, max_iter=60,
             et_start=1, fmt="int8", soft=False, layers=-1, iters=8),
        # The paper's multi-edge ensemble (1568 x 1600 base matrix, Z = 625)
        # above its waterfall.
        dict(name="multi_edge", kind="decode", code="met", Z=625, frames=16, snr=0.032, max_iter=200,
             et_start=1, fmt="fp32", soft=False, layers=-1, iters=65),
        # Row-layered decoding, the schedule the autotuner picks at this SNR.
        dict(name="layered", kind="decode", code="r002", Z=20000, frames=16, snr=0.13, max_iter=30,
             et_start=1, fmt="fp32", soft=False, layers=0, iters=6),
        # Frames of nine codes in one batched decode, FP16 messages.
        dict(name="mixed_codes", kind="multi", frames=4, max_iter=100, fmt="fp16", iters=6),
        # Serving: frames loaded into a pool, stepped to their end, collected.
        dict(name="pool", kind="pool", code="r005", Z=5000, frames=24, slots=32, snr=0.5, max_iter=12,
             passes=4, fmt="fp16", layers=-1, iters=12),
    ]


def _log_int(rng, lo, hi) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    """A case of the listed ranges: any code family, lifting sizes that give
    n = 1,600 to 10^6 (odd ones too), 1 to 64 frames of at most 16 * 10^6 bits
    together, every message format and schedule."""
    kind = rng.choice(["maps", "decode", "decode", "decode", "soft", "layered", "alice", "multi", "pool"])
    fmt = rng.choice(["fp32", "fp32", "fp16", "int8"])
    if kind == "multi":
        return dict(kind="multi", frames=rng.randint(1, 6), max_iter=_log_int(rng, 5, 100), fmt=fmt, iters=6)
    code = rng.choice(["r002", "r002", "r005", "r010", "met"])
    nb = BASE[code][1]
    Z = _log_int(rng, 8 if code == "met" else 64, 1000000 // nb)
    n = nb * Z
    frames = _log_int(rng, 1, max(1, min(64, 16000000 // n)))
    snr = {"r002": rng.choice([0.029, 0.13, 0.16, 0.2]), "r005": rng.choice([0.1, 0.5]),
           "r010": rng.choice([0.2, 1.0]), "met": rng.choice([0.029, 0.032, 0.036])}[code]
    if kind in ("maps", "alice"):  # whole 8-blocks and words in every frame
        Z = max(32, Z // 32 * 32)
    if kind == "maps":
        return dict(kind="maps", code=code, Z=Z, frames=frames, snr=snr, d=rng.choice([1, 2, 4, 8, 8]))
    if kind == "pool":
        return dict(kind="pool", code=code, Z=Z, frames=frames, slots=frames + rng.randint(0, 8), snr=snr,
                    max_iter=rng.randint(4, 20), passes=rng.randint(1, 8), fmt=fmt,
                    layers=rng.choice([-1, -1, 2]), iters=10)
    if kind == "layered":
        layers = rng.choice([0, 2, 7]) if code != "met" else rng.choice([2, 7, 64])
        max_iter = rng.randint(2, 30)
        return dict(kind="decode", code=code, Z=Z, frames=frames, snr=snr, max_iter=max_iter, et_start=1,
                    fmt=fmt, soft=False, layers=layers, iters=max_iter)
    if kind == "soft":
        max_iter = rng.randint(1, 50)
        return dict(kind="decode", code=code, Z=Z, frames=frames, snr=snr, max_iter=max_iter,
                    et_start=max_iter + 1, fmt=fmt, soft=True, layers=-1, iters=max_iter)
    max_iter = _log_int(rng, 5, 300 if code == "met" else 500)
    return dict(kind=kind, code=code, Z=Z, frames=frames, snr=snr, max_iter=max_iter,
                et_start=rng.choice([1, 1, max_iter // 2 + 1]), fmt=fmt, soft=False, layers=-1, iters=max_iter)


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=32)
def _base(code: str, Z: int) -> dict:
    return CODES[code](Z)


def _words(bits: torch.Tensor) -> torch.Tensor:
    """0/1 [F, n] -> packed int32 [F, ceil(n / 32)], least significant bit first."""
    F, n = bits.shape
    nw = (n + 31) // 32
    pad = torch.zeros((F, nw * 32), dtype=torch.int64, device=bits.device)
    pad[:, :n] = bits
    w = (pad.view(F, nw, 32) << torch.arange(32, device=bits.device)).sum(-1)
    return torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32)


def _edges(base: dict, dev):
    """(base row, flat variable index [E, Z]) of every circulant."""
    Z = base["Z"]
    row = torch.as_tensor(base["row"], dtype=torch.int64, device=dev)
    col = torch.as_tensor(base["col"], dtype=torch.int64, device=dev)
    shift = torch.as_tensor(base["shift"], dtype=torch.int64, device=dev)
    i = torch.arange(Z, device=dev)
    return row, col[:, None] * Z + (i[None, :] + shift[:, None]) % Z


def _syndrome(base: dict, bits: torch.Tensor) -> torch.Tensor:
    """0/1 [F, n] -> 0/1 [F, m], m = mb Z."""
    row, var = _edges(base, bits.device)
    F = bits.shape[0]
    out = []
    for f in range(F):
        s = torch.zeros((base["mb"], base["Z"]), dtype=torch.int32, device=bits.device)
        s.index_add_(0, row, bits[f][var].to(torch.int32))
        out.append((s & 1).reshape(1, -1))
    return torch.cat(out)


def _mul(a: torch.Tensor, b: torch.Tensor) -> torch.Tensor:
    """Cayley-Dickson product over the last dimension (1, 2, 4 or 8):
    (p, q)(r, s) = (p r - conj(s) q, s p + q conj(r))."""
    d = a.shape[-1]
    if d == 1:
        return a * b
    p, qq, r, s = a[..., :d // 2], a[..., d // 2:], b[..., :d // 2], b[..., d // 2:]
    return torch.cat([_mul(p, r) - _mul(_conj(s), qq), _mul(s, p) + _mul(qq, _conj(r))], -1)


def _conj(a: torch.Tensor) -> torch.Tensor:
    return torch.cat([a[..., :1], -a[..., 1:]], -1)


def _frames(code: str, Z: int, F: int, snr: float, seed: int) -> dict:
    """Bits, syndrome words and the channel draws of F frames."""
    base = _base(code, Z)
    n = base["nb"] * Z
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    bits = torch.randint(0, 2, (F, n), generator=g, device="cuda", dtype=torch.int8)
    x = torch.randn(F * n, generator=g, device="cuda")
    y = x + torch.randn(F * n, generator=g, device="cuda") * (1.0 / snr) ** 0.5
    return dict(base=base, n=n, bits=bits, x=x, y=y, g=g)


def _message(f: dict, d: int) -> torch.Tensor:
    u = (1.0 - 2.0 * f["bits"].to(torch.float32)).view(-1, d)
    return _mul(u, f["y"].view(-1, d)).reshape(-1)


def _llrs(code: str, Z: int, F: int, snr: float, seed: int):
    """(LLRs float[F n] as the 8-dimensional map gives them, syndrome words):
    blocks of eight bits share |X|^2 ~ chi^2_8, and Q = (snr |X|^2 / 4)(U + N)
    with N ~ N(0, 8 / (snr |X|^2))."""
    f = _frames(code, Z, F, snr, seed)
    n = f["n"]
    pad = -(F * n) % 8
    x2 = torch.cat([f["x"], f["x"][:pad]]).view(-1, 8).pow(2).sum(-1)
    x2 = x2.repeat_interleave(8)[:F * n]
    u = 1.0 - 2.0 * f["bits"].to(torch.float32).view(-1)
    noise = torch.randn(F * n, generator=f["g"], device="cuda")
    llr = 0.25 * snr * x2 * u + (0.5 * snr * x2).sqrt() * noise
    return llr, _words(_syndrome(f["base"], f["bits"])).view(-1)


def _code(code: str, Z: int):
    return q.create_code_from(_base(code, Z))


def _params(case: dict):
    p = q.qcldpc_params_init(msg_format=FMT[case["fmt"]], et_start=case.get("et_start", 1))
    if case.get("layers", -1) >= 0:
        p.schedule, p.layers = 1, case["layers"]
    return p


def prepare(case: dict, seed: int) -> dict:
    kind, s = case["kind"], dict(case=case)
    if kind == "multi":
        s["codes"] = [_code(c, Z) for c, Z in MIX]
        s["n_frames"] = [case["frames"] + (i % 2) for i in range(len(MIX))]
        s["llr"], s["syn"] = [], []
        for i, (c, Z) in enumerate(MIX):
            llr, syn = _llrs(c, Z, s["n_frames"][i], MIX_SNR[c], seed * 16 + i)
            s["llr"].append(llr)
            s["syn"].append(syn)
        s["dec"] = q.MultiDecoder(s["codes"], s["n_frames"], _params(case))
        return s
    code = _code(case["code"], case["Z"])
    s["code"] = code
    F, n = case["frames"], code.n
    if kind == "maps":
        f = _frames(case["code"], case["Z"], F, case["snr"], seed)
        s.update(x=f["x"], y=f["y"], bits=_words(f["bits"]).view(-1))
        s["msg"], s["llr"] = torch.empty_like(f["x"]), torch.empty_like(f["x"])
        s["syn"] = torch.empty(F * ((code.m + 31) // 32), dtype=torch.int32, device="cuda")
        return s
    if kind == "alice":
        f = _frames(case["code"], case["Z"], F, case["snr"], seed)
        s.update(x=f["x"], msg=_message(f, 8), llr=torch.empty_like(f["x"]),
                 syn=_words(_syndrome(f["base"], f["bits"])).view(-1))
    else:
        s["llr"], s["syn"] = _llrs(case["code"], case["Z"], F, case["snr"], seed)
    if kind == "pool":
        s["pool"] = q.Pool(code, case["slots"], case["max_iter"], _params(case))
        s["slots"] = torch.arange(case["slots"] - F, case["slots"], dtype=torch.int32, device="cuda")
        s["out"] = (torch.empty(F * ((code.k + 31) // 32), dtype=torch.int32, device="cuda"),
                    torch.empty(F, dtype=torch.int32, device="cuda"),
                    torch.empty(F, dtype=torch.int32, device="cuda"))
        return s
    s["dec"] = q.Decoder(code, F, _params(case), soft=case["soft"])
    return s


def run(s: dict):
    case = s["case"]
    kind = case["kind"]
    if kind == "maps":
        n, d = s["x"].numel(), case["d"]
        q.qcldpc_bob_message(d, s["y"], s["bits"], n, s["msg"])
        q.qcldpc_syndrome(s["code"], s["bits"], s["syn"], case["frames"])
        q.qcldpc_llr(d, s["x"], s["msg"], n, case["snr"], s["llr"])
        return {"msg": s["msg"], "syn": s["syn"], "llr": s["llr"]}
    if kind == "multi":
        s["dec"].decode(s["llr"], s["syn"], case["max_iter"])
        return {"keys": s["dec"].keys, "converged": s["dec"].converged, "iters": s["dec"].iters}
    if kind == "pool":
        keys, conv, iters = s["out"]
        q.qcldpc_pool_load(s["pool"], case["frames"], s["slots"], s["llr"], s["syn"])
        # every frame has stopped after max_iter + 1 passes
        for _ in range(-(-(case["max_iter"] + 1) // case["passes"])):
            q.qcldpc_pool_step(s["pool"], case["passes"])
        q.qcldpc_pool_collect(s["pool"], case["frames"], s["slots"], keys, conv, iters)
        return {"keys": keys, "converged": conv, "iters": iters}
    if kind == "alice":
        q.qcldpc_llr_8d(s["x"], s["msg"], s["x"].numel(), case["snr"], s["llr"])
    s["dec"].decode(s["llr"], s["syn"], case["max_iter"])
    out = {"keys": s["dec"].keys, "converged": s["dec"].converged, "iters": s["dec"].iters}
    if case["soft"]:
        out["posterior"] = s["dec"].posterior
    return out


# ------------------------------------------------------------ reference side

def work(case: dict) -> dict:
    """Inputs read once and outputs written once; operations: 23 per bit of an
    8-dimensional product (15 d / 8 for the others), and per iteration 60 per
    heavy edge (two evaluations of Phi and the sums), 6 per degree-1 edge."""
    def decode(code, Z, F, iters, soft=False):
        mb, nb, nh, nd1 = BASE[code]
        n, m = nb * Z, mb * Z
        return (F * (4 * n + m / 8 + (n - m) / 8 + 8 + (4 * n if soft else 0)),
                F * iters * Z * (60.0 * nh + 6.0 * nd1))

    kind = case["kind"]
    if kind == "multi":
        parts = [decode(c, Z, case["frames"] + (i % 2), min(case["iters"], case["max_iter"]))
                 for i, (c, Z) in enumerate(MIX)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    mb, nb, nh, nd1 = BASE[case["code"]]
    bits = case["frames"] * nb * case["Z"]
    if kind == "maps":
        # y, bits -> M; bits -> syndrome; x, M -> LLRs
        return {"bytes": bits * (4 + 4 + 1 / 8 + 4 + 4) + case["frames"] * mb * case["Z"] / 8,
                "flops": 2.0 * bits * 15 * case["d"] / 8}
    b, f = decode(case["code"], case["Z"], case["frames"], min(case["iters"], case["max_iter"]),
                  case.get("soft", False))
    if kind == "alice":
        b, f = b + 8 * bits, f + 15.0 * bits
    return {"bytes": b, "flops": f}


def _phi(x: torch.Tensor) -> torch.Tensor:
    return torch.log1p(2.0 / torch.expm1(x))


def _flood64(base: dict, llr: torch.Tensor, syn: torch.Tensor, iters: int,
             clip: float = 15.0, floor: float = 1e-6) -> torch.Tensor:
    """Posteriors of one frame after `iters` flooding iterations, float64."""
    Z, mb = base["Z"], base["mb"]
    row, var = _edges(base, llr.device)
    Q = llr.double()
    sgn_s = 1.0 - 2.0 * syn.view(mb, Z).double()
    m = torch.zeros(var.shape, dtype=torch.float64, device=llr.device)
    L = Q
    for _ in range(iters):
        v = (L[var] - m).clamp(-clip, clip)
        neg = (v < 0)
        a = _phi(v.abs().clamp(min=floor))
        tot = torch.zeros((mb, Z), dtype=torch.float64, device=llr.device).index_add_(0, row, a)
        par = torch.zeros((mb, Z), dtype=torch.int32, device=llr.device)
        par.index_add_(0, row, neg.to(torch.int32))
        odd = (par[row] - neg.to(torch.int32)) & 1
        mag = _phi((tot[row] - a).clamp(min=floor))
        m = ((1.0 - 2.0 * odd) * sgn_s[row] * mag).clamp(-clip, clip)
        L = Q.clone().index_add_(0, var.reshape(-1), m.reshape(-1))
    return L


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "maps":
        f = _frames(case["code"], case["Z"], case["frames"], case["snr"], seed)
        d = case["d"]
        f["y"] = f["y"].double()
        u = (1.0 - 2.0 * f["bits"].double()).view(-1, d)
        msg = _mul(u, f["y"].view(-1, d))
        llr = _mul(msg, _conj(f["x"].double().view(-1, d))) * (2.0 * case["snr"] / d)
        return {"msg": msg.reshape(-1), "syn": None, "llr": llr.reshape(-1)}
    if kind == "decode" and case["soft"] and case["fmt"] == "fp32":
        if case["frames"] * work(case)["flops"] > 4e12:
            return None
        base = _base(case["code"], case["Z"])
        F, m = case["frames"], base["mb"] * case["Z"]
        llr, syn = _llrs(case["code"], case["Z"], F, case["snr"], seed)
        sh = torch.arange(32, device=syn.device, dtype=torch.int32)
        sbits = ((syn.view(F, -1)[:, :, None] >> sh) & 1).view(F, -1)[:, :m]
        post = [_flood64(base, llr.view(F, -1)[f], sbits[f], case["max_iter"]) for f in range(F)]
        return {"keys": None, "converged": None, "iters": None, "posterior": torch.cat(post)}
    return None
