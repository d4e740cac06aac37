"""Timing cases: the decoding, training and serving work a program gives this library.

Every case goes through the package's public Python entry points.  Inputs are made here
with plain torch (systematic BCH encoding, BPSK over AWGN, LLR = 2y/sigma^2, uniform
random automorphisms), from the seed alone and independent of the library's kernels;
only the parity-check matrix comes from the library's own code object, as the plan a
program keeps.  ``exact`` restates the decoders and the training gradient in FP64.

Families
  hybrid  enhanced NMS with OSD on the failed frames, device buffers, kept workspace
  sweep   one point of an FER curve: simulate frames, draw automorphisms, decode, count
  plain   single min-sum decoder on the standard matrix (no automorphisms, no OSD)
  osd     order-p OSD alone on every frame
  train   forward, loss and backward of the normalization factors (torch.autograd)
  host    frames in pinned host memory through the host pipeline
  serve   a burst of mixed requests through the continuous-batching server
"""
import functools
import math

import numpy as np
import torch

from paper_2412_20828_gb300 import autograd as AG
from paper_2412_20828_gb300 import bchdec as B

ALPHA = 0.78
SERVE_CODES = ((63, 45), (127, 99))
PRIM = {15: 0b10011, 63: 0b1000011, 127: 0b10001001}
CODES = {63: (36, 45), 127: (64, 78, 99)}


def listed():
    return [
        # a client's single small request: a handful of frames, where launches and the
        # latency of one frame's iterations are all there is
        {"name": "request_63_45_f7", "kind": "hybrid", "n": 63, "k": 45, "frames": 7,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "fp32", "soft": False, "ld": 64},
        # a mid-size request of the long code that also wants the soft output
        {"name": "request_127_99_f1531", "kind": "hybrid", "n": 127, "k": 99, "frames": 1531,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "fp32", "soft": True, "ld": 128},
        # the largest request of the serving workload (1 to 4096 frames)
        {"name": "request_63_36_f4096", "kind": "hybrid", "n": 63, "k": 36, "frames": 4096,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "fp32", "soft": False, "ld": 64},
        # bulk decoding of the short code over the whole Eb/N0 grid: the main workload
        {"name": "batch_63_36", "kind": "hybrid", "n": 63, "k": 36, "frames": 3_000_000,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "fp32", "soft": False, "ld": 64},
        # one point of an error-rate curve, frames simulated on the device
        {"name": "sweep_63_45", "kind": "sweep", "n": 63, "k": 45, "frames": 1_000_000,
         "lo": 3.0, "hi": 3.0, "iters": 12, "P": 3, "msg": "fp32", "soft": False, "ld": 64},
        # bulk decoding of the long low-rate code (rows of weight 24, OSD on many frames)
        {"name": "batch_127_64", "kind": "hybrid", "n": 127, "k": 64, "frames": 200_001,
         "lo": 2.0, "hi": 5.0, "iters": 12, "P": 3, "msg": "fp32", "soft": False, "ld": 128},
        # messages stored in binary16
        {"name": "fp16_63_36", "kind": "hybrid", "n": 63, "k": 36, "frames": 1_000_003,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "fp16", "soft": False, "ld": 64},
        # 8-bit messages with fractional bits and rescaling (the form within 0.1 dB)
        {"name": "int8_63_45", "kind": "hybrid", "n": 63, "k": 45, "frames": 700_001,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "int8", "soft": False, "ld": 64},
        # the classical decoder the paper starts from
        {"name": "plain_63_36", "kind": "plain", "n": 63, "k": 36, "frames": 10_000,
         "lo": 3.0, "hi": 3.0, "iters": 8, "ld": 64},
        # one training step of the per-iteration factors at the workload's batch size
        {"name": "train_127_64", "kind": "train", "n": 127, "k": 64, "frames": 65_536,
         "lo": 2.0, "hi": 5.0, "iters": 12, "P": 3, "ld": 128},
        # frames that live in pinned host memory, results returned there
        {"name": "host_63_45", "kind": "host", "n": 63, "k": 45, "frames": 400_000,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3, "msg": "fp32", "ld": 64},
        # a burst of mixed requests, sizes log-uniform as the serving workload has them
        {"name": "serve_burst", "kind": "serve", "requests": 96, "max_frames": 4096,
         "lo": 1.0, "hi": 6.0, "iters": 12, "P": 3},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hybrid"] * 6 + ["sweep", "plain", "osd", "train", "train", "host", "serve"])
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(8, 128), "max_frames": _log_uniform(rng, 64, 4096),
                "lo": 1.0, "hi": round(rng.uniform(3.0, 6.0), 2), "iters": 12, "P": 3}
    n = rng.choice([63, 63, 127])
    k = rng.choice(CODES[n])
    lo = round(rng.uniform(1.0, 4.0), 2)
    c = {"kind": kind, "n": n, "k": k, "frames": 0, "lo": lo, "hi": round(lo + rng.uniform(0.0, 2.5), 2),
         "iters": 12, "ld": rng.choice([n + 1, n + 1, n])}
    if kind == "hybrid":
        c["frames"] = _log_uniform(rng, 1, 1_500_000 if n == 63 else 150_000)
        c["msg"] = rng.choice(["fp32", "fp32", "fp32", "fp16", "int8"])
        # three random automorphisms, or the paper's block of nine with few iterations
        c["P"], c["iters"] = rng.choice([(3, 12), (3, 12), (3, 8), (9, 4)])
        c["soft"] = c["msg"] == "fp32" and c["frames"] <= 20_000 and rng.random() < 0.5
    elif kind == "sweep":
        c["frames"] = _log_uniform(rng, 10_000, 1_000_000 if n == 63 else 100_000)
        c.update(msg="fp32", P=3, soft=False, hi=lo)
    elif kind == "plain":
        c["frames"] = _log_uniform(rng, 100, 200_000 if n == 63 else 50_000)
        c["iters"] = rng.choice([4, 8, 10])
    elif kind == "osd":
        c["frames"] = _log_uniform(rng, 10, 200_000 if n == 63 else 20_000)
        c["order"] = rng.choice([1, 2, 2])
    elif kind == "train":
        c["frames"] = _log_uniform(rng, 256, 65_536)
        c["iters"], c["P"] = rng.choice([4, 8, 12]), 3
    else:
        c["frames"] = _log_uniform(rng, 1_000, 600_000 if n == 63 else 60_000)
        c.update(msg="fp32", P=3)
    return c


# ---------------------------------------------------------------- what a program keeps
@functools.lru_cache(maxsize=None)
def _code(n, k):
    return B.Code(n, k)


@functools.lru_cache(maxsize=None)
def _std(n, k):
    return B.Code(n, k, kind=B.PCM_STANDARD)


@functools.lru_cache(maxsize=None)
def _server():
    # an idle kernel leaves the GPU after 0.3 ms, for programs that share it
    return B.Server([_code(*c) for c in SERVE_CODES], [_std(*c) for c in SERVE_CODES], 12, ALPHA,
                    n_autos=3, osd_order=2, budget_bytes=1 << 30, max_requests=512,
                    max_frames_per_request=4096, idle_exit_us=300)


def _params(case):
    kw = {"fp32": {}, "fp16": {"msg": B.MSG_FP16}, "int8": {"msg": B.MSG_INT8, "rescale": True, "qfrac": 8}}
    return B.params(case["iters"], ALPHA, n_autos=case["P"], osd_order=2, **kw[case["msg"]])


# ---------------------------------------------------------------- inputs (plain torch)
@functools.lru_cache(maxsize=None)
def _parity(n, k):
    """Parity part of every unit message of the systematic narrow-sense BCH code, [k][n-k]."""
    m = n.bit_length()
    exp = [1]
    for _ in range(n - 1):
        v = exp[-1] << 1
        exp.append(v ^ PRIM[n] if v >> m else v)
    log = {v: i for i, v in enumerate(exp)}

    def times(a, b):
        return exp[(log[a] + log[b]) % n] if a and b else 0

    g, used, s = [1], set(), 1
    while len(g) - 1 < n - k:
        if s not in used:
            coset = {s * 2 ** j % n for j in range(m)}
            used |= coset
            for e in sorted(coset):  # g *= (x + alpha^e)
                g = [(g[i - 1] if i else 0) ^ (times(g[i], exp[e]) if i < len(g) else 0)
                     for i in range(len(g) + 1)]
        s += 2
    gen = sum(c << i for i, c in enumerate(g))
    out = np.zeros((k, n - k), np.float32)
    for i in range(k):
        r = 1 << (n - k + i)
        while r.bit_length() > n - k:
            r ^= gen << (r.bit_length() - gen.bit_length())
        out[i] = [(r >> b) & 1 for b in range(n - k)]
    return out


def _pack(bits):
    F, n = bits.shape
    words = torch.zeros((F, (n + 63) // 64), dtype=torch.int64, device=bits.device)
    for i in range(n):
        words[:, i // 64] |= bits[:, i].to(torch.int64) << (i % 64)
    return words


def _frames(n, k, F, lo, hi, ld, gen):
    """(codewords [F][n] as 0/1 floats, LLRs [F][ld]) of F random frames, Eb/N0 U[lo, hi] dB."""
    dev = "cuda"
    msg = torch.randint(0, 2, (F, k), generator=gen, device=dev).float()
    bits = torch.cat([(msg @ torch.from_numpy(_parity(n, k)).to(dev)).round() % 2, msg], 1)
    ebn0 = lo + (hi - lo) * torch.rand((F, 1), generator=gen, device=dev)
    s2 = n / (2.0 * k * 10.0 ** (ebn0 / 10.0))
    llr = torch.zeros((F, ld), device=dev)
    llr[:, :n] = (1 - 2 * bits + s2.sqrt() * torch.randn((F, n), generator=gen, device=dev)) * (2 / s2)
    return bits, llr


def _autos(n, F, P, gen):
    """P distinct automorphisms per frame, s | j << 8, as int16 [F][P]."""
    m = n.bit_length()
    pick = torch.randint(0, n * m, (F, P), generator=gen, device="cuda")
    for p in range(1, P):  # redraw by stepping past the ones already taken
        for _ in range(p):
            clash = (pick[:, :p] == pick[:, p:p + 1]).any(1)
            pick[:, p] = torch.where(clash, (pick[:, p] + 1) % (n * m), pick[:, p])
    return (pick % n | (pick // n) << 8).to(torch.int16)


def _outputs(F, n, soft, ld):
    o = {"hard": torch.zeros((F, (n + 63) // 64), dtype=torch.int64, device="cuda"),
         "iters": torch.zeros(F, dtype=torch.uint8, device="cuda"),
         "flags": torch.zeros(F, dtype=torch.uint8, device="cuda")}
    if soft:
        o["llr_out"] = torch.zeros((F, ld), device="cuda")
    return o


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case, "seed": seed}
    if case["kind"] == "serve":
        s["srv"], s["reqs"] = _server(), []
        rng = np.random.default_rng(case["requests"])  # the burst's codes and sizes
        for i in range(case["requests"]):
            c = int(rng.integers(0, len(SERVE_CODES)))
            n, k = SERVE_CODES[c]
            F = int(round(math.exp(rng.uniform(0.0, math.log(case["max_frames"])))))
            _, llr = _frames(n, k, F, case["lo"], case["hi"], n + 1, gen)
            s["reqs"].append((c, llr.cpu().pin_memory(), seed + i, 1000 * i))
        return s
    n, k, F, ld = case["n"], case["k"], case["frames"], case["ld"]
    code, std = _code(n, k), _std(n, k)
    s.update(code=code, std=std)
    if case["kind"] == "sweep":
        s["p"] = _params(case)
        s["llr"] = torch.zeros((F, ld), device="cuda")
        s["autos"] = torch.zeros((F, case["P"]), dtype=torch.int16, device="cuda")
        s["cw"] = torch.zeros((F, (n + 63) // 64), dtype=torch.int64, device="cuda")
        s["out"] = _outputs(F, n, False, ld)
        s["ws"] = B.workspace(code, s["p"], F)
        return s
    bits, llr = _frames(n, k, F, case["lo"], case["hi"], ld, gen)
    if case["kind"] == "hybrid":
        s["p"] = _params(case)
        s["llr"], s["autos"] = llr, _autos(n, F, case["P"], gen)
        s["out"] = _outputs(F, n, case["soft"], ld)
        s["ws"] = B.workspace(code, s["p"], F)
        code.kernel_info(s["p"].msg, case["P"])
    elif case["kind"] == "plain":
        s["p"] = B.params(case["iters"], ALPHA, n_autos=0)
        s["llr"], s["out"] = llr, _outputs(F, n, True, ld)
        s["ws"] = B.workspace(std, s["p"], F)
    elif case["kind"] == "osd":
        s["llr"], s["out"] = llr, _outputs(F, n, False, ld)
        s["list"] = torch.arange(F, dtype=torch.int32, device="cuda")
        s["count"] = torch.full((1,), F, dtype=torch.int32, device="cuda")
        s["ws"] = torch.zeros(256, dtype=torch.uint8, device="cuda")
    elif case["kind"] == "train":
        s["llr"], s["autos"], s["cw"] = llr, _autos(n, F, case["P"], gen), _pack(bits)
        s["alpha"] = torch.full((case["iters"],), 0.7, device="cuda")
    elif case["kind"] == "host":
        s["p"] = _params(case)
        s["dec"] = B.HostDecoder(code, std, s["p"], ld, chunk_frames=1 << 20)
        s["llr"] = llr.cpu().pin_memory()
        s["out"] = {"hard": torch.zeros((F, (n + 63) // 64), dtype=torch.int64).pin_memory(),
                    "iters": torch.zeros(F, dtype=torch.uint8).pin_memory(),
                    "flags": torch.zeros(F, dtype=torch.uint8).pin_memory()}
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s["case"]["kind"]
    if kind == "serve":
        return _run_serve(s)
    if kind == "train":
        return _run_train(s)
    if kind == "host":
        o = s["out"]
        s["dec"].run(s["llr"], s["seed"], 0, o["hard"], o["iters"], o["flags"])
        return o
    if kind == "osd":
        o = s["out"]
        B.osd_decode(s["std"], s["case"]["order"], s["llr"], s["list"], s["count"], o["hard"], ws=s["ws"])
        return o["hard"]
    o = s["out"]
    if kind == "plain":
        B.nms_decode(s["std"], s["p"], s["llr"], None, o["hard"], o["iters"], o["flags"], o["llr_out"],
                     ws=s["ws"])
        return o
    if kind == "sweep":
        c = s["case"]
        B.gen_frames(s["code"], c["lo"], c["hi"], s["seed"], 0, s["llr"], s["cw"])
        B.draw_automorphisms(c["n"], c["P"], s["seed"] + 1, 0, s["autos"])
    B.hybrid_decode(s["code"], s["std"], s["p"], s["llr"], s["autos"], o["hard"], o["iters"], o["flags"],
                    llr_out=o.get("llr_out"), ws=s["ws"])
    if kind == "sweep":
        counters = torch.zeros(8, dtype=torch.int64, device="cuda")
        B.count_errors(s["case"]["n"], o["hard"], s["cw"], o["iters"], o["flags"], counters)
        return {"counters": counters, "llr": s["llr"], "codeword": s["cw"], **o}
    return o


def _run_train(s):
    llr = s["llr"].detach().requires_grad_(True)
    alpha = s["alpha"].detach().requires_grad_(True)
    y = AG.enhanced_nms(llr, alpha, s["code"], s["autos"])
    loss = AG.bce(y, s["cw"], s["code"])
    loss.backward()
    n = s["case"]["n"]
    return {"y": y.detach()[:, :n], "loss": loss.detach(), "grad_llr": llr.grad[:, :n],
            "grad_alpha": alpha.grad}


def _run_serve(s):
    srv = s["srv"]
    rids = [srv.submit(*r) for r in s["reqs"]]
    left, got = set(rids), {}
    while left:
        for rid in srv.poll(timeout_us=1000):
            if rid in left:
                got[rid] = srv.fetch(rid)
                left.discard(rid)
    out = {}
    for c in range(len(SERVE_CODES)):
        mine = [got[rid] for rid, r in zip(rids, s["reqs"]) if r[0] == c]
        if mine:
            out["code%d" % c] = [np.concatenate(x) for x in zip(*mine)]
    return out


# ---------------------------------------------------------------- the least a pass must do
# mean iterations of enhanced NMS (limit 12, P = 3) at Eb/N0 = 1.0, 1.5, ... 6.0 dB
MEAN_ITERS = {
    (63, 36): (9.6, 8.4, 6.9, 5.3, 3.8, 2.7, 1.8, 1.4, 1.1, 1.0, 1.0),
    (63, 45): (6.1, 5.1, 4.1, 3.1, 2.2, 1.6, 1.3, 1.1, 1.0, 1.0, 1.0),
    (127, 64): (11.9, 11.7, 11.2, 10.3, 8.6, 6.5, 4.4, 2.7, 1.8, 1.3, 1.1),
    (127, 78): (11.9, 11.6, 10.9, 9.7, 7.8, 5.5, 3.5, 2.1, 1.4, 1.1, 1.0),
    (127, 99): (11.9, 11.7, 11.2, 10.2, 8.6, 6.4, 4.3, 2.6, 1.6, 1.2, 1.1),
}


def _mean_iters(case):
    at = np.linspace(case["lo"], case["hi"], 16)
    mean = np.interp(at, 1.0 + 0.5 * np.arange(11), MEAN_ITERS[case["n"], case["k"]]).mean()
    return 1.0 + (mean - 1.0) * (case["iters"] - 1) / 11


# edges of the optimized and the standard matrices
EDGES = {(63, 36): (850, 486), (63, 45): (576, 432), (127, 64): (2890, 2142), (127, 78): (2744, 2156),
         (127, 99): (2464, 1344)}


def work(case):
    """Bytes: inputs read and outputs written once.  flops: 8 lane operations per edge update
    (two smallest magnitudes, sign, select, accumulate, gather); OSD: its weight-2 patterns
    are pruned, so only the elimination's row operations count."""
    if case["kind"] == "serve":
        F = case["requests"] * case["max_frames"] / (2 * math.log(case["max_frames"]))  # per code
        b = f = 0.0
        for n, k in SERVE_CODES:
            w = work({**case, "kind": "host", "n": n, "k": k, "frames": F})
            b, f = b + w["bytes"], f + w["flops"]
        return {"bytes": b, "flops": f}
    n, k, F = case["n"], case["k"], case["frames"]
    W = 8 * ((n + 63) // 64)
    opt, std = EDGES[n, k]
    if case["kind"] == "plain":
        return {"bytes": F * (8 * n + W + 2), "flops": F * std * case["iters"] * 8}
    if case["kind"] == "osd":
        return {"bytes": F * (4 * n + W + 4), "flops": F * n * (n - k)}
    P = case["P"]
    if case["kind"] == "train":  # checkpoints written and read, LLRs in, y and gradients out
        I = case["iters"]
        return {"bytes": F * n * 4 * (2 * I + 4), "flops": F * opt * P * I * 8 * 3}
    b = F * (4 * n + 2 * P + W + 2)
    if case.get("soft"):
        b += F * 4 * n
    if case["kind"] == "sweep":
        b += F * (4 * n + 2 * W)
    return {"bytes": b, "flops": F * opt * P * _mean_iters(case) * 8}


# ---------------------------------------------------------------- FP64 restatements
def _index(H):
    """Columns of every row, padded with n (a column of neutral values)."""
    n = H.shape[1]
    w = int(H.sum(1).max())
    idx = np.full((H.shape[0], w), n, np.int64)
    for r, row in enumerate(H):
        c = np.flatnonzero(row)
        idx[r, :len(c)] = c
    return torch.from_numpy(idx).cuda()


def _positions(n, autos):
    """pi(i) = 2^j i + s mod n for every frame and map: [F][P][n]."""
    a = autos.to(torch.int64) & 0xffff
    i = torch.arange(n, device=a.device)
    return ((1 << (a >> 8)).unsqueeze(-1) * i + (a & 0xff).unsqueeze(-1)) % n


def _row_stats(z, idx):
    """Per row: magnitudes with their two smallest, and signs without the edge's own."""
    return _edge_stats(torch.cat([z, torch.full_like(z[:, :1], math.inf)], 1)[:, idx])


def _edge_stats(e):
    mag = e.abs()
    m1, at = mag.min(2, keepdim=True)
    m2, at2 = mag.scatter(2, at, math.inf).min(2, keepdim=True)
    two, at = torch.cat([m1, m2], 2), torch.cat([at, at2], 2)
    sg = torch.where(e < 0, -1.0, 1.0)
    return mag, two, at, sg * sg.prod(2, keepdim=True)


def _c2v(z, idx, alpha):
    mag, two, at, sg = _row_stats(z, idx)
    m = torch.where(mag == two[..., :1], two[..., 1:], two[..., :1])
    return torch.where(torch.isinf(mag), 0.0, alpha * sg * m)


def _columns(v, idx, n):
    out = torch.zeros((v.shape[0], n + 1), dtype=v.dtype, device=v.device)
    out.index_add_(1, idx.reshape(-1), v.reshape(v.shape[0], -1))
    return out[:, :n]


def _step(y, pos, idx, alpha):
    """One merged iteration of Algorithm 1 (reading A): y + mean over the maps of the c2v sums."""
    n = y.shape[1]
    add = torch.zeros_like(y)
    for p in range(pos.shape[1]):
        z = torch.empty_like(y).scatter_(1, pos[:, p], y)
        add += _columns(_c2v(z, idx, alpha), idx, n).gather(1, pos[:, p])
    return y + add / pos.shape[1]


def _nms64(H, llr, autos, iters):
    n = H.shape[1]
    idx, Ht = _index(H), torch.from_numpy(H.T.astype(np.float64)).cuda()
    y, live = llr[:, :n].double().clone(), torch.arange(llr.shape[0], device=llr.device)
    for _ in range(iters):
        y[live] = _step(y[live], _positions(n, autos[live]), idx, ALPHA32)
        bad = ((y[live] < 0).double() @ Ht % 2 > 0.5).any(1)
        live = live[bad]
        if not live.numel():
            break
    return y


def _plain64(H, llr, iters):
    n = H.shape[1]
    idx, Ht = _index(H), torch.from_numpy(H.T.astype(np.float64)).cuda()
    L = llr[:, :n].double()
    x, live = L.clone(), torch.arange(llr.shape[0], device=llr.device)
    c = torch.zeros((llr.shape[0],) + tuple(idx.shape), dtype=torch.float64, device=llr.device)
    for _ in range(iters):
        pad = torch.cat([x[live], torch.full_like(x[live][:, :1], math.inf)], 1)
        e = pad[:, idx] - c[live]
        mag, two, _, sg = _edge_stats(e)
        m = torch.where(mag == two[..., :1], two[..., 1:], two[..., :1])
        c[live] = torch.where(torch.isinf(mag), 0.0, ALPHA32 * sg * m)
        x[live] = L[live] + _columns(c[live], idx, n)
        live = live[((x[live] < 0).double() @ Ht % 2 > 0.5).any(1)]
        if not live.numel():
            break
    return x


ALPHA32 = float(np.float32(ALPHA))


def _train64(H, llr, autos, bits, iters, total):
    """y, summed loss and the gradients of one chunk of a batch of `total` frames."""
    n, idx = H.shape[1], _index(H)
    al = float(np.float32(0.7))
    pos, ys = _positions(n, autos), [llr[:, :n].double()]
    for _ in range(iters):
        ys.append(_step(ys[-1], pos, idx, al))
    sgn = 1 - 2 * bits.double()
    x = -sgn * ys[-1]
    loss = torch.nn.functional.softplus(x, threshold=1e4).sum() / (total * n)
    g = torch.sigmoid(x) * -sgn / (total * n)
    P, da = pos.shape[1], torch.zeros(iters, dtype=torch.float64, device=llr.device)
    for t in range(iters - 1, -1, -1):
        new = g.clone()
        for p in range(P):
            z = torch.empty_like(g).scatter_(1, pos[:, p], ys[t])
            gz = torch.zeros_like(g).scatter_(1, pos[:, p], g) / P
            mag, two, at, sg = _row_stats(z, idx)
            ge = torch.cat([gz, torch.zeros_like(gz[:, :1])], 1)[:, idx] * sg
            slot = torch.arange(idx.shape[1], device=idx.device)
            first = slot == at[..., :1]
            da[t] += (ge * torch.where(first, two[..., 1:], two[..., :1])).sum()
            other = (ge * ~first).sum(2, keepdim=True)
            own = (ge * first).sum(2, keepdim=True)
            ez = torch.cat([z, torch.zeros_like(z[:, :1])], 1)[:, idx]
            sz = torch.where(ez < 0, -1.0, 1.0)
            d = al * sz * torch.where(first, other, torch.where(slot == at[..., 1:], own, 0.0))
            new += _columns(d, idx, n).gather(1, pos[:, p])
        g = new
    return ys[-1], loss, g, da


def _mix32(a, b):
    """(high, low) words of the 64-bit product of a constant and 32-bit words in int64."""
    lo = (a & 0xffff) * b
    hi = (a >> 16) * b + (lo >> 16)
    return hi >> 16, ((hi & 0xffff) << 16) | (lo & 0xffff)


def _philox(c, key):
    k0, k1 = key
    c = list(c)
    for r in range(10):
        h0, l0 = _mix32(0xD2511F53, c[0])
        h1, l1 = _mix32(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xffffffff, (k1 + 0xBB67AE85) & 0xffffffff
    return c


def _sim64(n, k, F, ebn0, seed, ld):
    """The library's simulated LLRs (its documented Philox4x32-10 addressing) in FP64."""
    f = torch.arange(F, dtype=torch.int64, device="cuda").unsqueeze(1)
    zero, key = torch.zeros_like(f), (seed & 0xffffffff, seed >> 32)
    mw = torch.cat(_philox((f, zero, zero, zero), key), 1)
    at = torch.arange(k, device="cuda")
    msg = ((mw[:, at // 32] >> (at % 32)) & 1).float()
    bits = torch.cat([(msg @ torch.from_numpy(_parity(n, k)).cuda()).round() % 2, msg], 1).double()
    b = torch.arange((n + 3) // 4, dtype=torch.int64, device="cuda").unsqueeze(0) + zero
    u = [((w >> 8).double() + 0.5) / 2 ** 24 for w in _philox((f + 0 * b, 0 * b, b, 0 * b + 1), key)]
    z = []
    for i in (0, 2):
        r, th = (-2 * u[i].log()).sqrt(), 2 * math.pi * u[i + 1]
        z += [r * th.cos(), r * th.sin()]
    z = torch.stack(z, 2).reshape(F, -1)[:, :n]
    s2 = n / (2.0 * k * 10.0 ** (ebn0 / 10.0))
    out = torch.zeros((F, ld), dtype=torch.float64, device="cuda")
    out[:, :n] = (1 - 2 * bits + math.sqrt(s2) * z) * (2 / s2)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return {"llr": _sim64(case["n"], case["k"], case["frames"], case["lo"], seed, case["ld"])}
    if kind not in ("hybrid", "plain", "train") or (kind == "hybrid" and not case["soft"]):
        return None  # whole numbers only
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, k, F, ld = case["n"], case["k"], case["frames"], case["ld"]
    bits, llr = _frames(n, k, F, case["lo"], case["hi"], ld, gen)
    step = 2048
    parts = range(0, F, step)
    if kind == "plain":
        H = _std(n, k).dense()
        y = torch.cat([_plain64(H, llr[i:i + step], case["iters"]) for i in parts])
    else:
        H, autos = _code(n, k).dense(), _autos(n, F, case["P"], gen)
        if kind == "train":
            got = [_train64(H, llr[i:i + step], autos[i:i + step], bits[i:i + step], case["iters"], F)
                   for i in parts]
            return {"y": torch.cat([g[0] for g in got]), "loss": sum(g[1] for g in got),
                    "grad_llr": torch.cat([g[2] for g in got]), "grad_alpha": sum(g[3] for g in got)}
        y = torch.cat([_nms64(H, llr[i:i + step], autos[i:i + step], case["iters"]) for i in parts])
    out = torch.zeros((F, ld), dtype=torch.float64, device="cuda")
    out[:, :n] = y
    return {"llr_out": out}
