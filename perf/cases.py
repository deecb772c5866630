"""What this framework is used for, as cases that can be timed.

A case is a dict of plain values. The kinds:

* ``decode``: one ``ldpc_decode`` of a batch of frames that is on the GPU;
* ``host``: ``ldpc_decode_host_stream`` on batches in pinned host memory;
* ``batch``: ``ldpc_batch_run`` over several codes;
* ``chain``: one batch of the BER simulator, from the information bits or the
  all-zero word through channel and decoder to the error counts;
* ``encode_ira`` and ``encode_dense``: codewords from information words.

Codes are named as in ``ber.CODES``; ``ira<n>`` is the rate-1/2 IRA code of the
sweep over lengths and ``qc<n>`` its quasi-cyclic (4, 8)-regular counterpart.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1609_01567_gb300 import ber, inputs, ldpc, mixed, sweep

L_MAX = 20.0

# Eb/N0 (dB) from which nearly every frame of a code decodes within 50
# iterations; the draws start a little above it.
WATERFALL_DB = {"n1008": 2.2, "n64800": 1.2, **mixed.EBN0_AT_FER_1E2}
SWEEP_DB = 2.2  # the rate-1/2 codes of the sweep over lengths

# Mean flooding passes of an early-exit decode, for the work it cannot do without.
MEAN_PASSES = 12


def listed():
    return [
        # A receive chain that decodes frames as they arrive: one short frame,
        # stopped at its first zero syndrome. Launches and latency.
        {"name": "one_frame_n1008", "kind": "decode", "code": "n1008", "frames": 1, "ebn0": 2.0, "max_iter": 50,
         "early": True, "msg": "f32", "post": True},
        # The small batch: 1000 short frames, soft output wanted.
        {"name": "batch_n1008_f1000", "kind": "decode", "code": "n1008", "frames": 1000, "ebn0": 2.0, "max_iter": 50,
         "early": True, "msg": "f32", "post": True},
        # A mid-length code with a few nodes of high degree, fixed iterations.
        {"name": "wide_n8192_f256_bf16", "kind": "decode", "code": "n8192_r3/4_deg64_96", "frames": 256, "ebn0": 3.0,
         "max_iter": 10, "early": False, "msg": "bf16", "post": False},
        # Offset min-sum on a low-rate code, a ragged number of frames.
        {"name": "min_sum_n16200_f301", "kind": "decode", "code": "n16200_r1/3", "frames": 301, "ebn0": 1.6,
         "max_iter": 50, "early": True, "msg": "f32", "post": True, "rule": "min_sum", "beta": 0.15},
        # The benchmark's workload: the long code, ten fixed iterations.
        {"name": "long_n64800_f256", "kind": "decode", "code": "n64800", "frames": 256, "ebn0": 1.0, "max_iter": 10,
         "early": False, "msg": "f32", "post": False},
        # The same code decoded until its frames stop, half-precision messages.
        {"name": "long_n64800_f256_stop_f16", "kind": "decode", "code": "n64800", "frames": 256, "ebn0": 1.6,
         "max_iter": 50, "early": True, "msg": "f16", "post": False},
        # A high-rate long code with the smallest messages, a ragged batch.
        {"name": "rate56_n64800_f165_i8", "kind": "decode", "code": "n64800_r5/6", "frames": 165, "ebn0": 3.2,
         "max_iter": 50, "early": True, "msg": "i8", "post": False},
        # The paper's benchmark form: 10,000 codewords at 2 dB, channel noise,
        # decoder and error count on one stream.
        {"name": "simulate_qc2048_f10000", "kind": "chain", "code": "qc2048", "frames": 10000, "ebn0": 2.0,
         "max_iter": 50, "msg": "f32", "words": "zero"},
        # Many codes at once: 4096 frames over eight codes, one graph.
        {"name": "mixed_8_codes_f4096", "kind": "batch", "codes": ";".join(c[2] for c in inputs.MIXED_SPECS),
         "frames": ";".join(map(str, inputs.zipf_frames(mixed.TOTAL_FRAMES, len(inputs.MIXED_SPECS)))),
         "margin": 0.0, "max_iter": 50, "msg": "bf16"},
        # End to end: batches in host memory, copies in and out.
        {"name": "host_n64800_4x256", "kind": "host", "code": "n64800", "frames": 256, "batches": 4, "ebn0": 1.0,
         "max_iter": 10, "early": False, "msg": "f32"},
        # The transmit side: the long staircase code, and a lifted code
        # without a staircase through the dense encoder.
        {"name": "encode_n64800_f1024", "kind": "encode_ira", "code": "n64800", "frames": 1024},
        {"name": "encode_qc8192_f1000", "kind": "encode_dense", "code": "qc8192", "frames": 1000},
    ]


def draw(rng):
    kind = rng.choices(("decode", "chain", "batch", "host", "encode_ira", "encode_dense"), (11, 3, 1, 1, 2, 2))[0]

    def spread(lo, hi):  # log-uniform whole number
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def length(hi):  # a multiple of 8, not only powers of two
        return 8 * spread(32, hi // 8)

    def named():
        return rng.choice(("n1008", "n64800") + tuple(s[2] for s in inputs.MIXED_SPECS))

    if kind == "encode_dense":
        code = "qc%d" % length(8192)
        return {"kind": kind, "code": code, "frames": spread(1, min(10000, 40_000_000 // _n(code)))}
    if kind == "encode_ira":
        code = named() if rng.random() < 0.5 else "ira%d" % length(65536)
        return {"kind": kind, "code": code, "frames": spread(1, min(10000, 80_000_000 // _n(code)))}
    if kind == "batch":
        codes = [named() for _ in range(rng.randint(2, 6))]
        frames = [spread(1, min(1500, 9_000_000 // _n(c))) for c in codes]
        return {"kind": kind, "codes": ";".join(codes), "frames": ";".join(map(str, frames)),
                "margin": round(rng.uniform(0.1, 0.6), 3), "max_iter": 50, "msg": rng.choice(("f32", "f16", "bf16"))}
    code = rng.choice((named, lambda: "qc%d" % length(65536), lambda: "ira%d" % length(65536)))()
    case = {"kind": kind, "code": code, "frames": spread(1, max(1, min(10000, 20_000_000 // _n(code)))),
            "ebn0": round(WATERFALL_DB.get(code, SWEEP_DB) + rng.uniform(0.1, 0.8), 3),
            "max_iter": rng.choice((10, 20, 50)), "early": rng.random() < 0.7,
            "msg": rng.choice(("f32", "f32", "f16", "bf16", "i8"))}
    if kind == "chain":
        del case["early"]
        case["words"] = "zero" if code.startswith("qc") else rng.choice(("zero", "random"))
    elif kind == "host":
        case["batches"] = rng.randint(1, 4)
        case["frames"] = max(1, case["frames"] // case["batches"])
    else:
        case["post"] = rng.random() < 0.5
        if rng.random() < 0.25:
            case["rule"] = "min_sum"
            case["beta"] = rng.choice((0.0, 0.15, 0.3))
    return case


# ---------------------------------------------------------------------------
# codes, and the handles a program keeps
# ---------------------------------------------------------------------------

def _n(name):
    if name in ("n1008", "n64800"):
        return int(name[1:])
    for n, _k, spec in inputs.MIXED_SPECS:
        if spec == name:
            return n
    return int(name.removeprefix("qc").removeprefix("ira"))


@functools.lru_cache(maxsize=64)
def _code(name):
    if name in ber.CODES:
        return ber.CODES[name]()
    if name.startswith("qc"):
        return inputs.qc_stand_in_code(int(name[2:]))[0]
    return sweep.stand_in_code(int(name[3:]))


@functools.lru_cache(maxsize=12)
def _handle(name):
    if name.startswith("qc"):
        n = int(name[2:])
        return ldpc.ldpc_code_create_qc(4, 8, n // 8, inputs.qc_stand_in_code(n)[1])
    return ldpc.code_from_inputs(_code(name))


@functools.lru_cache(maxsize=16)
def _h1(name):
    """Rows and columns of the edges of the information bits, on the GPU."""
    c = _code(name)
    sel = c.cols < c.k
    return (torch.from_numpy(c.rows[sel].astype(np.int64)).cuda(), torch.from_numpy(c.cols[sel].astype(np.int64)).cuda())


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed, part=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + part)
    return g


def _words(name, info):
    """Codewords [F, n] (uint8) of a staircase code: p = running xor of H1 u."""
    c = _code(name)
    rows, cols = _h1(name)
    out = torch.empty((info.shape[0], c.n), dtype=torch.uint8, device=info.device)
    out[:, :c.k] = info
    step = max(1, 100_000_000 // max(1, rows.numel()))
    for f in range(0, info.shape[0], step):
        u = info[f:f + step]
        s = torch.zeros((c.m, u.shape[0]), dtype=torch.int32, device=u.device)
        s.index_add_(0, rows, u.t().contiguous()[cols].to(torch.int32))
        out[f:f + step, c.k:] = (s.cumsum(0) & 1).t().to(torch.uint8)
    return out


def _llr(name, frames, ebn0, gen):
    """Channel LLRs of noisy frames of random codewords. The lifted codes hold
    every word that is constant on the Z columns of each base column and has an
    even number of ones over a row's eight base columns."""
    c = _code(name)
    s2 = inputs.sigma2_from_ebn0(ebn0, c.rate)
    y = torch.randn((frames, c.n), generator=gen, device="cuda") * math.sqrt(s2)
    if c.k >= 0:
        info = torch.randint(0, 2, (frames, c.k), generator=gen, device="cuda", dtype=torch.uint8)
        y += 2.0 * _words(name, info).float() - 1.0
    else:
        blocks = torch.randint(0, 2, (frames, 7), generator=gen, device="cuda")
        blocks = torch.cat([blocks, blocks.sum(1, keepdim=True) & 1], 1)
        y += 2.0 * blocks.repeat_interleave(c.n // 8, 1).float() - 1.0
    return y * (2.0 / s2)


def _split(case):
    codes, frames = case["codes"].split(";"), [int(f) for f in case["frames"].split(";")]
    return list(zip(codes, frames))


def _inputs(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_llr(c, f, WATERFALL_DB[c] + case["margin"], _generator(seed, i))
                for i, (c, f) in enumerate(_split(case))]
    if kind == "host":
        return [_llr(case["code"], case["frames"], case["ebn0"], _generator(seed, i)) for i in range(case["batches"])]
    return _llr(case["code"], case["frames"], case["ebn0"], _generator(seed))


def _k(name):
    """Information bits of the word that the encoders take."""
    c = _code(name)
    return c.k if c.k >= 0 else ldpc.ldpc_code_build_encoder(_handle(name))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "batch":
        items = _split(case)
        s["llr"] = _inputs(case, seed)
        s["batch"] = ldpc.ldpc_batch_create([_handle(c) for c, _ in items], [f for _, f in items], case["max_iter"],
                                            msg_dtype=case["msg"])
        ldpc.ldpc_batch_tune(s["batch"], s["llr"])
        s["out"] = [{"bits": torch.zeros((f, _n(c)), dtype=torch.uint8, device="cuda"),
                     "iters": torch.zeros((f,), dtype=torch.int32, device="cuda"),
                     "ok": torch.zeros((f,), dtype=torch.uint8, device="cuda")} for c, f in items]
        return s
    name, frames = case["code"], case["frames"]
    s["code"] = _handle(name)
    if kind == "host":
        s["llr"] = [x.cpu().pin_memory() for x in _inputs(case, seed)]
        s["out"] = [{"bits": torch.zeros((frames, _n(name)), dtype=torch.uint8, pin_memory=True),
                     "iters": torch.zeros((frames,), dtype=torch.int32, pin_memory=True),
                     "ok": torch.zeros((frames,), dtype=torch.uint8, pin_memory=True)} for _ in s["llr"]]
        return s
    cuda = functools.partial(torch.zeros, device="cuda")
    if kind in ("encode_ira", "encode_dense"):
        s["info"] = torch.randint(0, 2, (frames, _k(name)), generator=_generator(seed), device="cuda",
                                  dtype=torch.uint8)
        s["words"] = cuda((frames, _n(name)), dtype=torch.uint8)
        return s
    s["out"] = {"bits": cuda((frames, _n(name)), dtype=torch.uint8), "iters": cuda((frames,), dtype=torch.int32),
                "ok": cuda((frames,), dtype=torch.uint8)}
    if kind == "chain":
        s["seed"] = int(seed)
        s["sigma2"] = inputs.sigma2_from_ebn0(case["ebn0"], _code(name).rate)
        s["llr"] = cuda((frames, _n(name)))
        if case["words"] == "random":
            s["info"] = cuda((frames, _k(name)), dtype=torch.uint8)
            s["words"] = cuda((frames, _n(name)), dtype=torch.uint8)
        return s
    if case["post"]:
        s["out"]["post"] = cuda((frames, _n(name)))
    s["llr"] = _inputs(case, seed)
    return s


def _rule(case):
    return {"rule": case.get("rule", "sum_product"), "rule_beta": case.get("beta", 0.0)}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "decode":
        return ldpc.ldpc_decode(s["code"], s["llr"], case["max_iter"], early_exit=case["early"], msg_dtype=case["msg"],
                                want_post=case["post"], out=s["out"], **_rule(case))
    if kind == "batch":
        return ldpc.ldpc_batch_run(s["batch"], s["llr"], s["out"])
    if kind == "host":
        return ldpc.ldpc_decode_host_stream(s["code"], s["llr"], case["max_iter"], early_exit=case["early"],
                                            msg_dtype=case["msg"], outs=s["out"])
    if kind == "encode_ira":
        return ldpc.ldpc_encode_ira(s["code"], s["info"], out=s["words"])
    if kind == "encode_dense":
        return ldpc.ldpc_encode(s["code"], s["info"], out=s["words"])
    # one batch of the BER simulator
    words = None
    frames, n = s["llr"].shape
    if case["words"] == "random":
        ldpc.ldpc_gen_bits(s["seed"], 0, frames, s["info"].shape[1], out=s["info"])
        words = ldpc.ldpc_encode_ira(s["code"], s["info"], out=s["words"])
    ldpc.ldpc_gen_awgn(s["seed"], 0, frames, n, s["sigma2"], words, out=s["llr"])
    out = ldpc.ldpc_decode(s["code"], s["llr"], case["max_iter"], msg_dtype=case["msg"], want_post=False, out=s["out"])
    counts = ldpc.ldpc_count_errors(out["bits"], words, out["iters"], out["ok"])
    result = {"llr": s["llr"], "bits": out["bits"], "iters": out["iters"], "ok": out["ok"], "counts": counts}
    return dict(result, words=words) if words is not None else result


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def _decode_work(name, frames, case):
    c = _code(name)
    passes = MEAN_PASSES if case.get("early", True) else case["max_iter"] + 1
    passes = min(passes, case["max_iter"] + 1)
    # a check output takes about 30 operations an edge, a posterior one
    return {"bytes": frames * (c.n * (5 + (4 if case.get("post") else 0)) + 5) + 8 * c.n_edges,
            "flops": 31 * frames * c.n_edges * passes}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_decode_work(c, f, case) for c, f in _split(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    name, frames = case["code"], case["frames"]
    c = _code(name)
    if kind in ("encode_ira", "encode_dense"):
        k = c.k if c.k >= 0 else c.n - c.m
        return {"bytes": frames * (k + c.n), "flops": frames * c.n_edges}
    w = _decode_work(name, frames, case)
    if kind == "host":
        return {k: v * case["batches"] for k, v in w.items()}
    if kind == "chain":  # the LLRs are written too; about 100 operations a sample
        w["bytes"] += frames * c.n * 4
        w["flops"] += frames * c.n * 100
    return w


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _phi(x):
    return torch.log1p(2.0 / torch.expm1(x))


def _rounded(r, msg):
    if msg == "f16":
        return r.to(torch.float16).to(torch.float64)
    if msg == "bf16":
        return r.to(torch.bfloat16).to(torch.float64)
    if msg == "i8":
        return torch.round(r * (127.0 / 20.0)).clamp(-127, 127) * (20.0 / 127.0)
    return r


def _check_rule(q, rule, beta):
    """New messages of checks of one degree: q [checks, degree, F]."""
    others_odd = ((q > 0).sum(1, keepdim=True) - (q > 0).long()) & 1
    if rule == "min_sum":
        x = q.abs().clamp(max=L_MAX)
        if q.shape[1] == 1:
            m = torch.full_like(x, L_MAX)
        else:
            two, at = x.topk(2, dim=1, largest=False)
            pos = torch.arange(q.shape[1], device=q.device)[None, :, None]
            m = torch.where(pos == at[:, :1], two[:, 1:], two[:, :1])
        mag = (m - beta).clamp(0.0, L_MAX)
    else:
        low = math.log1p(2.0 / math.expm1(L_MAX))
        p = _phi(q.abs().clamp(low, L_MAX))
        zero = torch.zeros_like(p[:, :1])
        before = torch.cat([zero, p[:, :-1]], 1).cumsum(1)
        after = torch.cat([p[:, 1:], zero], 1).flip(1).cumsum(1).flip(1)
        mag = _phi((before + after).clamp(low, L_MAX))
    return torch.where(others_odd.bool(), mag, -mag)


def _posteriors(name, llr, case):
    """Posteriors [F, n] of the flooding decoder (Algorithm 2) in 64 bits."""
    c = _code(name)
    order = np.lexsort((c.cols, c.rows))
    degree = np.bincount(c.rows, minlength=c.m)
    first = np.concatenate([[0], np.cumsum(degree)])
    groups = [torch.from_numpy(c.cols[order][first[:-1][degree == d][:, None] + np.arange(d)].astype(np.int64)).cuda()
              for d in np.unique(degree[degree > 0])]
    rule, beta = case.get("rule", "sum_product"), case.get("beta", 0.0)
    out = []
    for part in llr.split(max(1, 60_000_000 // c.n_edges)):
        lam = part.double().t().contiguous()
        app = lam.clone()
        r = [torch.zeros((), dtype=torch.float64, device="cuda")] * len(groups)
        done = torch.zeros(lam.shape[1], dtype=torch.bool, device="cuda")
        for _ in range(case["max_iter"] + 1):
            new = lam.clone()
            for i, g in enumerate(groups):
                r[i] = _rounded(_check_rule(app[g] - r[i], rule, beta), case["msg"])
                new.index_add_(0, g.reshape(-1), r[i].reshape(-1, lam.shape[1]))
            app = torch.where(done, app, new)
            if case["early"]:
                odd = torch.zeros_like(done)
                for g in groups:
                    odd |= (((app[g] > 0).sum(1) & 1) != 0).any(0)
                done |= ~odd
                if bool(done.all()):
                    break
        out.append(app.t())
    return torch.cat(out)


def _philox(seed, key1, frames, blocks):
    """uint64 [F, 4 * blocks]: Philox-4x64-10 at counters (b, f), key (seed, key1)."""
    words = np.empty((frames, 4 * blocks), dtype=np.uint64)
    top = 2 ** 64 - 1
    for f in range(frames):  # numpy steps the counter before each block
        at = [top, f - 1, 0, 0] if f else [top] * 4
        words[f] = np.random.Philox(key=np.array([seed, key1], dtype=np.uint64),
                                    counter=np.array(at, dtype=np.uint64)).random_raw(4 * blocks)
    return words


def _channel(case, seed):
    """Channel LLRs [F, n] of the chain in 64 bits."""
    name, frames = case["code"], case["frames"]
    c = _code(name)
    x = -1.0
    if case["words"] == "random":
        bits = np.unpackbits(_philox(seed, 1, frames, -(-c.k // 256)).view(np.uint8), axis=1, bitorder="little")
        x = 2.0 * _words(name, torch.from_numpy(bits[:, :c.k].copy()).cuda()).double().cpu().numpy() - 1.0
    w = (_philox(seed, 0, frames, -(-c.n // 4)) >> np.uint64(40)).astype(np.float64)
    rho = np.sqrt(-2.0 * np.log((w[:, 0::2] + 1.0) * 2.0 ** -24))
    angle = 2.0 * np.pi * (w[:, 1::2] * 2.0 ** -24)
    z = np.stack([rho * np.cos(angle), rho * np.sin(angle)], axis=-1).reshape(frames, -1)[:, :c.n]
    s2 = float(np.float32(inputs.sigma2_from_ebn0(case["ebn0"], c.rate)))
    return torch.from_numpy(2.0 * (x + math.sqrt(s2) * z) / s2)


def exact(case, seed):
    if case["kind"] == "chain":
        out = {"llr": _channel(case, seed), "bits": None, "iters": None, "ok": None, "counts": None}
        return dict(out, words=None) if case["words"] == "random" else out
    if case["kind"] == "decode" and case["post"]:
        return {"bits": None, "iters": None, "ok": None,
                "post": _posteriors(case["code"], _inputs(case, seed), case)}
    return None  # decisions, counts and codewords: whole numbers
