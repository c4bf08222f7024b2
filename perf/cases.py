"""The measured workloads of the library: what a program that uses it has it do.

Kinds: ``sketch`` (B = Omega A), ``rsvd`` (Algorithm 1), ``nystrom``
(Algorithm 2, FP32 storage with FP64 arithmetic as the serving loop runs it)
and ``serve`` (a mixed batch through the serving loop).  Matrices follow the
library's own generators: a low-rank part with exponentially decaying singular
values (exp(-i / 10) in the small FP64 workload, else exp(-4 i / k), so that
the wanted triplets stand apart) plus Gaussian noise of spectral norm 0.003 of
the largest; PSD ones without the noise.

Factors: rSVD on FP32 and 16-bit data computes in FP32 and hands its factors
out in double.  A caller of such data keeps them in FP32 beside it, and so does
``run``; FP64 data and FP64 arithmetic keep the doubles.
"""

import math

import numpy as np
import torch

import paper_2210_11295_gb300 as bsrht

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}


def listed():
    return [
        # The small FP64 workload's sketch: one call, all latency and launches.
        {"name": "sketch_small_f64", "kind": "sketch", "dtype": "f64", "n": 4096, "m": 256, "p": 4, "l": 128},
        # An ordinary request of the mixed stream.
        {"name": "sketch_request_f32", "kind": "sketch", "dtype": "f32", "n": 65536, "m": 700, "p": 8, "l": 150},
        # A data set as it comes: no power of two, rows that end off 16 bytes.
        {"name": "sketch_ragged_f32", "kind": "sketch", "dtype": "f32", "n": 300007, "m": 1250, "p": 6, "l": 300},
        # The tall-skinny workload in FP32 (16 GiB), the headline sketch.
        {"name": "sketch_tall_f32", "kind": "sketch", "dtype": "f32", "n": 1 << 20, "m": 4096, "p": 4, "l": 512},
        # The same in the paper's arithmetic, FP64 (16 GiB: half the rows).
        {"name": "sketch_tall_f64", "kind": "sketch", "dtype": "f64", "n": 1 << 19, "m": 4096, "p": 4, "l": 512},
        # The 16-bit workload.
        {"name": "sketch_tall_bf16", "kind": "sketch", "dtype": "bf16", "n": 1 << 20, "m": 8192, "p": 8, "l": 1024},
        # The small FP64 workload: sketch and rank-20 rSVD.
        {"name": "rsvd_small_f64", "kind": "rsvd", "dtype": "f64", "n": 4096, "m": 256, "p": 4, "l": 128, "k": 20,
         "decay": 10},
        # FP64 at a size where the tall products weigh.
        {"name": "rsvd_mid_f64", "kind": "rsvd", "dtype": "f64", "n": 1 << 17, "m": 2048, "p": 8, "l": 256, "k": 64},
        # The headline rSVD.
        {"name": "rsvd_tall_f32", "kind": "rsvd", "dtype": "f32", "n": 1 << 20, "m": 4096, "p": 16, "l": 512, "k": 100},
        # A BF16 request of the mixed stream (half of its matrices are BF16).
        {"name": "rsvd_request_bf16", "kind": "rsvd", "dtype": "bf16", "n": 1 << 18, "m": 2000, "p": 8, "l": 400,
         "k": 100},
        # A Nystrom request of the mixed stream.
        {"name": "nystrom_request", "kind": "nystrom", "n": 1 << 14, "p": 16, "l": 400, "k": 100},
        # A batch of the mixed stream through the serving loop: sketches and rSVDs, FP32 and BF16.
        {"name": "serve_batch", "kind": "serve", "requests": 12, "log2n": 17, "stream": 5},
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["sketch", "sketch", "sketch", "rsvd", "rsvd", "nystrom", "serve"])
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(6, 12), "log2n": rng.randint(14, 17),
                "stream": rng.randint(6, 1 << 20)}
    if kind == "nystrom":
        l = log_uniform(64, 512)
        return {"kind": kind, "n": rng.randint(1 << 13, 1 << 14) // 16 * 16, "p": 16, "l": l, "k": max(1, l // 4)}
    dtype = rng.choice(["f64", "f32", "f32", "bf16"] if kind == "rsvd" else ["f64", "f32", "f32", "bf16", "f16"])
    # Half of the sizes as the generators give them, half as data sets come.
    m = log_uniform(64, 8192 if kind == "sketch" and dtype in ("bf16", "f16") else 4096)
    if rng.random() < 0.5:
        m = -(-m // 8) * 8
    most = (1 << 34) // (m * BYTES[dtype])
    if kind == "rsvd":
        l = min(log_uniform(64, 512), m)
        most = min(most, (1 << (36 if dtype == "f64" else 40)) // (m * l))
    else:
        l = log_uniform(64, 1024)
    n = log_uniform(4096, max(8192, min(1 << 20, most)))
    if rng.random() < 0.5:
        n = 1 << (n.bit_length() - 1)
    p = rng.choice([1, 2, 3, 4, 6, 8, 16] if kind == "sketch" else [4, 8, 16])
    case = {"kind": kind, "dtype": dtype, "n": n, "m": m, "p": p, "l": min(l, n)}
    if kind == "rsvd":
        case["k"] = max(1, min(100, case["l"] // 4))
    return case


# ------------------------------------------------------------------ inputs
def _lowrank(n, m, decay, dtype, gen, width=None):
    """n x m, sigma_i = exp(-i / decay), plus noise; `width`: columns of the buffer that holds it."""
    work = torch.float64 if dtype == torch.float64 else torch.float32
    rank = min(int(8 * decay), n, m)
    g1 = torch.randn(n, rank, generator=gen, device="cuda", dtype=torch.float32) / math.sqrt(n)
    g2 = torch.randn(m, rank, generator=gen, device="cuda", dtype=torch.float32) / math.sqrt(m)
    sigma = torch.exp(-1.0 / decay * torch.arange(1, rank + 1, device="cuda", dtype=torch.float32))
    g2t = (g2 * sigma).T.contiguous()
    buf = torch.zeros(n, width or m, device="cuda", dtype=dtype)
    step = max(1, (1 << 28) // m)
    for r0 in range(0, n, step):
        r1 = min(n, r0 + step)
        block = 0.003 / (math.sqrt(n) + math.sqrt(m)) * torch.randn(r1 - r0, m, generator=gen, device="cuda", dtype=work)
        block += g1[r0:r1] @ g2t
        buf[r0:r1, :m] = block
    return buf[:, :m]


def _psd(n, k, rank, gen):
    """Symmetric PSD n x n, lambda_i = exp(-2 i / k), FP32."""
    g = torch.randn(n, rank, generator=gen, device="cuda", dtype=torch.float32) / math.sqrt(n)
    lam = torch.exp(-2.0 / k * torch.arange(1, rank + 1, device="cuda", dtype=torch.float32))
    a = (g * lam) @ g.T
    return 0.5 * (a + a.T)


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _requests(case):
    """The shapes of a served batch, from the case alone."""
    rng = np.random.default_rng(case["stream"])
    out = []
    for i in range(case["requests"]):
        kind = "rsvd" if i % 4 == 3 else "sketch"
        dtype = str(rng.choice(["f32", "bf16"]))
        n = 1 << int(rng.integers(13, case["log2n"] + 1))
        m = int(round(math.exp(rng.uniform(math.log(64), math.log(1024)))))
        l = int(round(math.exp(rng.uniform(math.log(64), math.log(512)))))
        p = int(rng.choice([4, 8, 16]))
        l = min(l, m) if kind == "rsvd" else l
        out.append({"kind": kind, "dtype": dtype, "n": n, "m": m, "p": p, "l": l, "k": max(1, l // 4)})
    return out


def _request_input(q, gen):
    # Row stride as in a store of one matrix per size class: the next power of two of m.
    return _lowrank(q["n"], q["m"], q["k"] / 4, DTYPES[q["dtype"]], gen, 1 << (q["m"] - 1).bit_length())


def _inputs(case, seed):
    gen = _generator(seed)
    if case["kind"] == "serve":
        return [_request_input(q, gen) for q in _requests(case)]
    if case["kind"] == "nystrom":
        return _psd(case["n"], case["k"], min(case["n"], 5 * case["l"] // 4 + 16), gen)
    decay = case.get("decay") or case.get("k", max(1, case["l"] // 4)) / 4
    return _lowrank(case["n"], case["m"], decay, DTYPES[case["dtype"]], gen)


class _Served:
    """A server with its batch of requests and their output buffers."""

    def __init__(self, case, inputs, seed):
        self.seed, self.inputs, self.requests, self.outs = seed, inputs, _requests(case), []
        for q in self.requests:
            if q["kind"] == "sketch":
                self.outs.append((torch.empty(q["l"], q["m"], device="cuda", dtype=torch.float32),))
            else:
                n, m, k = q["n"], q["m"], q["k"]
                self.outs.append(tuple(torch.empty(s, device="cuda", dtype=torch.float64)
                                       for s in ((n, k), (k,), (m, k))))
        torch.cuda.synchronize()  # the server's streams are not ordered after this one
        self.server = bsrht.Server(4 << 30)

    def __del__(self):
        if getattr(self, "server", None) is not None:
            self.server.close()


def prepare(case, seed):
    a = _inputs(case, seed)
    if case["kind"] == "serve":
        return {"case": case, "served": _Served(case, a, seed)}
    return {"case": case, "a": a, "seed": int(seed)}


# -------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        return _run_served(state["served"])
    a, seed, p, l = state["a"], state["seed"], case["p"], case["l"]
    if case["kind"] == "sketch":
        return bsrht.bsrht_sketch(a, p, l, seed)
    if case["kind"] == "nystrom":
        u, lam = bsrht.bsrht_nystrom(a, case["k"], l, p, seed, precision=bsrht.PREC_F64)
        return {"u": u, "lam": lam}
    return _factors(bsrht.bsrht_rsvd(a, case["k"], l, p, seed), case["dtype"])


def _factors(usv, dtype):
    if dtype != "f64":
        usv = [x.float() for x in usv]
    return dict(zip(("u", "s", "v"), usv))


def _run_served(b):
    tickets = []
    for i, (q, a, out) in enumerate(zip(b.requests, b.inputs, b.outs)):
        if q["kind"] == "sketch":
            tickets.append(b.server.submit_sketch(a, q["p"], q["l"], b.seed + i, out[0]))
        else:
            tickets.append(b.server.submit_rsvd(a, q["k"], q["l"], q["p"], b.seed + i, out))
    for t in tickets:
        status = b.server.wait(t)
        if status != 0:
            raise RuntimeError(bsrht.strerror(status))
    return [out[0] if q["kind"] == "sketch" else _factors(out, q["dtype"]) for q, out in zip(b.requests, b.outs)]


# ------------------------------------------------------------------- work
def work(case):
    if case["kind"] == "serve":
        parts = [work(q) for q in _requests(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    l = case["l"]
    if case["kind"] == "nystrom":
        n, k = case["n"], case["k"]
        # A once, U and Lambda; the subsampled transform, Z and its Gram, U.
        return {"bytes": 4.0 * n * n + 8.0 * (n + 1) * k,
                "flops": n * n * math.log2(l) + 2.0 * n * l * l + n * l * l + 2.0 * n * l * k}
    n, m, es = case["n"], case["m"], BYTES[case["dtype"]]
    flops = n * m * math.log2(l)
    if case["kind"] == "sketch":
        return {"bytes": float(n * m * es + l * m * max(es, 4)), "flops": flops}
    k, fs = case["k"], 8 if case["dtype"] == "f64" else 4
    # The sketch, A Q, the Gram and the triangular factor of the tall QR, U.
    return {"bytes": float(n * m * es + fs * (n + m + 1) * k),
            "flops": flops + 2.0 * n * m * l + n * l * l + 2.0 * n * l * k}


# ------------------------------------------------------- exact, in 64 bits
def _mulhi(a, b):
    """High 64 bits of a * b (numpy uint64)."""
    mask, half = np.uint64(0xFFFFFFFF), np.uint64(32)
    a0, a1, b0, b1 = a & mask, a >> half, b & mask, b >> half
    low = a0 * b0
    mid = a1 * b0 + (low >> half)
    mid2 = a0 * b1 + (mid & mask)
    return a1 * b1 + (mid >> half) + (mid2 >> half)


def _philox(c0, c1, c2, seed):
    """Philox4x64-10 of the counters (c0, c1, c2, 0) with key (seed, 0): four words each."""
    x = [np.asarray(v, dtype=np.uint64) for v in np.broadcast_arrays(c0, c1, c2, 0)]
    m0, m1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    key = [int(seed) % (1 << 64), 0]
    for rnd in range(10):
        if rnd:
            key = [(key[0] + 0x9E3779B97F4A7C15) % (1 << 64), (key[1] + 0xBB67AE8584CAA73B) % (1 << 64)]
        with np.errstate(over="ignore"):
            x = [_mulhi(m1, x[2]) ^ x[1] ^ np.uint64(key[0]), m1 * x[2],
                 _mulhi(m0, x[0]) ^ x[3] ^ np.uint64(key[1]), m0 * x[0]]
    return np.stack(x, -1)


def _signs(count, block, stream, seed):
    """count signs (+-1) of one (block, stream): bit k & 63 of word (k >> 6) & 3 of counter k >> 8."""
    words = _philox(np.arange(-(-count // 256), dtype=np.uint64), block, stream, seed).reshape(-1)
    bits = (words[:, None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)
    return torch.from_numpy(1.0 - 2.0 * bits.reshape(-1)[:count].astype(np.float64)).cuda()


def _sketch64(a, p, l, seed):
    """Omega a in FP64: per block signs, the Walsh-Hadamard transform, the sampled rows, signs, the block sum."""
    n, m = a.shape
    rb = -(-n // p)
    r = 1 << max(0, (rb - 1).bit_length())
    rows = (_philox(np.arange(-(-l // 4), dtype=np.uint64), 0, 2, seed).reshape(-1)[:l] % np.uint64(r)).astype(np.int64)
    rows = torch.from_numpy(rows).cuda()
    out = torch.zeros(l, m, device="cuda", dtype=torch.float64)
    width = max(1, min(m, (1 << 28) // r))
    for i in range(p):
        d, dt = _signs(r, i, 0, seed), _signs(l, i, 1, seed)
        lo, hi = min(n, i * rb), min(n, (i + 1) * rb)
        for c0 in range(0, m, width):
            x = torch.zeros(r, min(width, m - c0), device="cuda", dtype=torch.float64)
            x[: hi - lo] = a[lo:hi, c0 : c0 + width].double() * d[: hi - lo, None]
            h = 1
            while h < r:
                v = x.view(r // (2 * h), 2, h, -1)
                s = v[:, 0] + v[:, 1]
                torch.sub(v[:, 0], v[:, 1], out=v[:, 1])
                v[:, 0] = s
                h *= 2
            out[:, c0 : c0 + width] += dt[:, None] * x[rows]
    return out / math.sqrt(l)


def _svd(x):
    """SVD of a small FP64 matrix by LAPACK."""
    u, s, vt = np.linalg.svd(x.cpu().numpy())
    return tuple(torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (u, s, vt.T))


def _positive(u, *others):
    """Each column of u with its largest entry positive; `others` get the same flips."""
    at = u.abs().argmax(0)
    flip = torch.sign(u[at, torch.arange(u.shape[1], device=u.device)])
    return [x * flip for x in (u, *others)]


def _rsvd64(a, k, l, p, seed):
    n = a.shape[0]
    y, r = torch.linalg.qr(_sketch64(a, p, l, seed).T.contiguous())
    ur, s, _ = _svd(r)
    q = y @ ur[:, : int((s > l * 2.0 ** -44 * s[0]).sum())]
    w = torch.empty(n, q.shape[1], device="cuda", dtype=torch.float64)
    for r0 in range(0, n, 1 << 16):
        w[r0 : r0 + (1 << 16)] = a[r0 : r0 + (1 << 16)].double() @ q
    t, r = torch.linalg.qr(w)
    us, s, vs = _svd(r)
    u, v = _positive(t @ us[:, :k], q @ vs[:, :k])
    return u, s[:k], v


def _nystrom64(a, k, l, p, seed):
    n = a.shape[0]
    omega = _sketch64(torch.eye(n, device="cuda", dtype=torch.float64), p, l, seed)
    y = _sketch64(a, p, l, seed).T
    nu = math.sqrt(n) * 2.0 ** -52 * float(torch.linalg.norm(y))
    y = y + nu * omega.T
    core = omega @ y
    c = torch.linalg.cholesky(0.5 * (core + core.T))
    z = torch.linalg.solve_triangular(c, y.T, upper=False).T.contiguous()
    t, r = torch.linalg.qr(z)
    us, s, _ = _svd(r)
    (u,) = _positive(t @ us[:, :k])
    return u, torch.clamp(s[:k] ** 2 - nu, min=0.0)


def exact(case, seed):
    a = _inputs(case, seed)
    todo = list(zip(_requests(case), a)) if case["kind"] == "serve" else [(case, a)]
    got = []
    for i, (q, x) in enumerate(todo):
        if q["kind"] == "sketch":
            got.append(_sketch64(x, q["p"], q["l"], seed + i))
        elif q["kind"] == "nystrom":
            got.append(dict(zip(("u", "lam"), _nystrom64(x, q["k"], q["l"], q["p"], seed + i))))
        else:
            got.append(dict(zip(("u", "s", "v"), _rsvd64(x, q["k"], q["l"], q["p"], seed + i))))
    return got if case["kind"] == "serve" else got[0]
