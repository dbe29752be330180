"""Measured cases: what a user of the library has it do, through the tensor-level
wrappers of ``paper_2609_11687_gb300.kashin``.

Four stages of the quantiser's life are covered, with the layer shapes of the synthetic
workloads in ``paper_2609_11687_gb300/synth.py``:

* ``quantise``    -- Algorithm 1 and the 2-bit coding of whole layers (``decompose`` for one
  matrix of a length, ``decompose_batch`` for several);
* ``product``     -- inference from the 2-bit planes: ``XP`` by ``apply_p_prepared`` on tables
  that ``prepare_p`` left at load time, then the product of every matrix of the layer with
  its activations (``matmul_2bit_batch`` for fp32, ``matmul_2bit_f16_batch`` for fp16 and
  bf16); one row is decode, hundreds are prefill;
* ``reconstruct`` and ``dequantise`` -- the load-time expansions to dense weights;
* ``rht``         -- the randomized-Hadamard pre-rotation of a layer's weights.

A case names its matrices as ``shapes``: ``"n:m,n:m,..."``, ``m`` vectors of length ``n``.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_11687_gb300 import kashin as kd
from paper_2609_11687_gb300 import synth

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}

# lengths with a compiled plan, and lengths of the run-time path that models have as widths
# or that the tests run
TUNED = (256, 512, 768, 1024, 1536, 2048, 3072, 4096, 8192, 11008, 14336, 16384)
RUNTIME = (640, 1000, 1280, 2560, 5120, 6144, 6912, 10000, 13824)


def _layer(specs):
    return ",".join(f"{s.N}:{s.M}" for s in specs)


OPT125M = _layer(synth.config2([0]))
LLAMA7B = _layer(synth.config3())


def listed():
    return [
        # a single small matrix: latency and launches, no full wave
        dict(name="quantise_256_f32", op="quantise", shapes="256:256", dtype="f32", layout="rows", iters=16, kmeans=0),
        # one small model's decoder layer: six matrices of two lengths, none of which fills the GPU
        dict(name="quantise_opt125m", op="quantise", shapes=OPT125M, dtype="f16", layout="rows", iters=16, kmeans=0),
        # the flagship: one 7B decoder layer, the step of the benchmark
        dict(name="quantise_llama7b", op="quantise", shapes=LLAMA7B, dtype="f16", layout="rows", iters=16, kmeans=0),
        # a model width without a compiled plan, in the paper's own layout (vector = column),
        # with the k-means refinement
        dict(name="quantise_5120_columns", op="quantise", shapes="5120:5120", dtype="bf16", layout="columns", iters=16,
             kmeans=3),
        # decode: one token through the 7B layer, full precision
        dict(name="decode_f32_b1", op="product", shapes=LLAMA7B, dtype="f32", batch=1),
        # a batch of sixteen sequences decoding in full precision
        dict(name="decode_f32_b16", op="product", shapes=LLAMA7B, dtype="f32", batch=16),
        # decode with 16-bit activations, four sequences
        dict(name="decode_f16_b4", op="product", shapes=LLAMA7B, dtype="f16", batch=4),
        # prefill: a prompt of 512 tokens through the 7B layer
        dict(name="prefill_f16_b512", op="product", shapes=LLAMA7B, dtype="f16", batch=512),
        # a short prompt of odd length through the small model's layer
        dict(name="prefill_bf16_b33", op="product", shapes=OPT125M, dtype="bf16", batch=33),
        # model load: dense weights of the 7B layer from codes and centres
        dict(name="reconstruct_llama7b", op="reconstruct", shapes=LLAMA7B, dtype="f16", layout="rows"),
        # model load for the folded product on dense factors: both planes of every matrix
        dict(name="dequantise_llama7b", op="dequantise", shapes=LLAMA7B, dtype="f16", layout="rows"),
        # the rotation before quantising (Kashin-DCT+H), the whole 7B layer
        dict(name="rht_llama7b", op="rht", shapes=LLAMA7B, dtype="f16", inverse=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_n(rng):
    kind = rng.random()
    if kind < 0.55:
        return rng.choice(TUNED)
    if kind < 0.8:
        return rng.choice(RUNTIME)
    while True:  # any other length with factors the run-time path takes
        n = rng.choice((3, 5, 7, 9, 11, 13, 15, 21, 25, 27, 35, 43, 45, 75)) * 2 ** rng.randint(3, 11)
        if 256 <= n <= 16384:
            return n


def draw(rng):
    op = rng.choice(("quantise", "quantise", "quantise", "product", "product", "product", "product", "reconstruct",
                     "dequantise", "rht"))
    n = _draw_n(rng)
    tuned = n in TUNED
    count = rng.randint(1, 4)
    iters = rng.choice((4, 8, 16, 16, 16, 32))
    # entries in all: no more than an eighth of the 7B layer's work (its blocks included
    # where the method iterates; the run-time lengths cost several times the compiled ones)
    most = 202e6 * (16 / iters / (8 if tuned else 12) if op == "quantise" else 0.25)
    ms = [_log_int(rng, 48, max(49, min(16384, most / count / n))) for _ in range(count)]
    shapes = ",".join(f"{n}:{m}" for m in ms)
    if op == "quantise":
        return dict(op=op, shapes=shapes, dtype=rng.choice(("f32", "f16", "f16", "bf16")),
                    layout=rng.choice(("rows", "rows", "columns")), iters=iters, kmeans=rng.choice((0, 0, 0, 1, 3)))
    if op == "product":
        dtype = rng.choice(("f32", "f16", "f16", "bf16"))
        return dict(op=op, shapes=shapes, dtype=dtype, batch=_log_int(rng, 1, 64 if dtype == "f32" else 512))
    if op == "rht":
        return dict(op=op, shapes=shapes, dtype=rng.choice(("f32", "f16", "bf16")), inverse=rng.random() < 0.3)
    return dict(op=op, shapes=shapes, dtype=rng.choice(("f32", "f16", "bf16")),
                layout=rng.choice(("rows", "rows", "columns")))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _shapes(case):
    return [tuple(int(v) for v in s.split(":")) for s in case["shapes"].split(",")]


def _groups(shapes):
    """Indices of the matrices of each vector length, in order of first appearance."""
    g = {}
    for i, (n, _) in enumerate(shapes):
        g.setdefault(n, []).append(i)
    return g


def _weights(case, seed, dtype):
    """Student-t weights with 0.1 % outlier input channels, vector-major (m, n)."""
    specs = [synth.MatrixSpec(f"w{i}", n, m, seed=1000 * int(seed) + i, std=0.015, dtype=dtype,
                              outlier_channel_frac=0.001, outlier_channel_scale=20.0)
             for i, (n, m) in enumerate(_shapes(case))]
    return [synth.generate(s, device="cuda") for s in specs], [s.sign_seed for s in specs]


def _coded(case, seed):
    """The layer's matrices as a user has them after quantisation: codes, centres, seeds."""
    ws, seeds = _weights(case, seed, torch.float16)
    decs = [None] * len(ws)
    for idx in _groups(_shapes(case)).values():
        for i, d in zip(idx, kd.decompose_batch([ws[i] for i in idx], 4, [seeds[i] for i in idx])):
            decs[i] = d
    return decs, seeds


def prepare(case, seed):
    shapes = _shapes(case)
    groups = _groups(shapes)
    st = dict(case=case, shapes=shapes, groups=groups)
    op = case["op"]
    if op in ("quantise", "rht"):
        ws, seeds = _weights(case, seed, DTYPES[case["dtype"]])
        if case.get("layout") == "columns":
            ws = [w.t().contiguous() for w in ws]
        st.update(ws=ws, seeds=seeds)
        if op == "quantise":
            st["workspaces"] = {n: kd.Workspace(n, count=len(idx)) for n, idx in groups.items()}
        else:
            st["outs"] = [torch.empty(w.shape, dtype=torch.float32, device="cuda") for w in ws]
        return st

    decs, seeds = _coded(case, seed)
    st.update(decs=decs, seeds=seeds)
    dt = DTYPES[case["dtype"]]
    if op == "product":
        b = case["batch"]
        g = torch.Generator(device="cuda").manual_seed(1000 * int(seed) + 999)
        total = sum(b * n for n, _ in shapes)
        flat = torch.randn(total, generator=g, device="cuda")
        flat.mul_(1.0 + 19.0 * (torch.rand(total, generator=g, device="cuda") < 0.001))  # outlier features

        def views(buf):
            out, at = [], 0
            for n, _ in shapes:
                out.append(buf[at:at + b * n].view(b, n))
                at += b * n
            return out

        x = flat.to(dt)
        st.update(x=x, xs=views(x), ys=[torch.empty((b, m), device="cuda") for _, m in shapes],
                  p={n: kd.prepare_p(n, [seeds[i] for i in idx]) for n, idx in groups.items()})
        xp32 = torch.empty(total, device="cuda")
        st.update(xp32=xp32, xps32=views(xp32))
        if dt == torch.float32:
            st.update(xs32=st["xs"], xps=st["xps32"])
        else:
            x32, xp = torch.empty(total, device="cuda"), torch.empty(total, dtype=dt, device="cuda")
            st.update(x32=x32, xs32=views(x32), xp=xp, xps=views(xp))
        return st

    cols = case["layout"] == "columns"

    def dense():
        return [torch.empty((n, m) if cols else (m, n), dtype=dt, device="cuda") for n, m in shapes]

    if op == "reconstruct":
        st.update(outs=dense(), workspaces={n: kd.Workspace(n, count=len(idx)) for n, idx in groups.items()})
    else:
        st.update(us=dense(), vs=dense())
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case, groups = st["case"], st["groups"]
    op = case["op"]
    if op == "quantise":
        res = [None] * len(st["ws"])
        for n, idx in groups.items():
            kw = dict(layout=case["layout"], workspace=st["workspaces"][n], kmeans_iters=case["kmeans"])
            if len(idx) == 1:
                ds = [kd.decompose(st["ws"][idx[0]], case["iters"], st["seeds"][idx[0]], **kw)]
            else:
                ds = kd.decompose_batch([st["ws"][i] for i in idx], case["iters"], [st["seeds"][i] for i in idx],
                                        coeffs=True, **kw)
            for i, d in zip(idx, ds):
                res[i] = [d.codes_u, d.codes_v, d.centres_u, d.centres_v, d.coeffs]
        return res
    if op == "product":
        half = case["dtype"] != "f32"
        if half:
            st["x32"].copy_(st["x"])
        for n, idx in groups.items():
            kd.apply_p_prepared([st["xs32"][i] for i in idx], st["p"][n], outs=[st["xps32"][i] for i in idx])
        if half:
            st["xp"].copy_(st["xp32"])
            return kd.matmul_2bit_f16_batch(st["decs"], st["xs"], st["xps"], outs=st["ys"])
        return kd.matmul_2bit_batch(st["decs"], st["xs"], st["xps"], outs=st["ys"])
    if op == "rht":
        return [kd.rht(w, s, inverse=case["inverse"], out=o) for w, s, o in zip(st["ws"], st["seeds"], st["outs"])]
    if op == "reconstruct":
        for n, idx in groups.items():
            kd.reconstruct_batch([st["decs"][i] for i in idx], n, [st["seeds"][i] for i in idx],
                                 dtype=DTYPES[case["dtype"]], layout=case["layout"], outs=[st["outs"][i] for i in idx],
                                 workspace=st["workspaces"][n])
        return st["outs"]
    for n, idx in groups.items():
        planes, outs = [], []
        for i in idx:
            d = st["decs"][i]
            planes += [(d.codes_u, d.centres_u), (d.codes_v, d.centres_v)]
            outs += [st["us"][i], st["vs"][i]]
        kd.dequantise_batch(planes, n, dtype=DTYPES[case["dtype"]], layout=case["layout"], outs=outs)
    return [st["us"], st["vs"]]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    esz = DTYPES[case["dtype"]].itemsize
    op = case["op"]
    nbytes = flops = 0.0
    for n, m in _shapes(case):
        coded = m * (2 * 4 * ((n + 15) // 16) + 2 * 16)  # both code planes and centre tables
        dct = 2.0 * n * math.log2(n)                     # one DCT of length n
        if op == "quantise":
            nbytes += esz * n * m + coded + 16 * m
            # per block: two P of two DCTs, 20 n for the four greedy steps; per refinement
            # step 3 compares and 7 adds per entry of each factor
            flops += m * (case["iters"] * (4 * dct + 20.0 * n) + case["kmeans"] * 2 * 10.0 * n)
        elif op == "product":
            b = case["batch"]
            nbytes += coded + b * (esz * n + 4 * m)
            flops += 2.0 * b * 2 * n * m + b * 2 * dct
        elif op == "reconstruct":
            nbytes += coded + esz * n * m
            flops += m * (2 * dct + n)
        elif op == "dequantise":
            nbytes += coded + 2 * esz * n * m
        else:
            b = _hadamard_block(n)
            nbytes += (esz + 4) * n * m
            flops += m * n * (math.log2(b) + 1)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _signs(seed, n):
    """+1 / -1 of a seeded sign set: bit 63 of SplitMix64 (Steele, Lea & Flood 2014) at
    seed + (j + 1) * 0x9E3779B97F4A7C15."""
    with np.errstate(over="ignore"):
        z = np.uint64(int(seed) & (2 ** 64 - 1)) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy(1.0 - 2.0 * (z >> np.uint64(63)).astype(np.float64)).cuda()


def _p64(x, eps):
    """IDCT(eps * DCT(x)) of the rows of a float64 tensor, through complex FFTs."""
    n = x.shape[1]
    h = (n + 1) // 2
    k = torch.arange(n, device=x.device, dtype=torch.float64)
    w = torch.polar(torch.ones_like(k), -math.pi * k / (2 * n))
    v = torch.cat([x[:, ::2], x[:, 1::2].flip(1)], dim=1)
    c = (torch.fft.fft(v) * w).real * eps
    mirror = torch.cat([torch.zeros_like(c[:, :1]), c[:, 1:].flip(1)], dim=1)
    v = torch.fft.ifft(torch.complex(c, -mirror) * w.conj()).real
    y = torch.empty_like(x)
    y[:, ::2] = v[:, :h]
    y[:, 1::2] = v[:, h:].flip(1)
    return y


def _quantise64(w, eps, iters, kmeans):
    """(centres_u, centres_v, coeffs) of the rows of w: Algorithm 1 (only its first block
    where no refinement follows) and the centres of both factors."""
    r = w.double()
    n = r.shape[1]
    x, u = r, torch.zeros_like(r)
    coeffs = []

    def step(r):
        lam = r.abs().sum(1, keepdim=True) / n
        d = torch.sign(r) * lam
        return d, r - d, lam

    for t in range(iters if kmeans else min(iters, 1)):
        for _ in range(2):
            d, r, lam = step(r)
            u = u + d
            if t == 0:
                coeffs.append(lam)
        r = _p64(r, eps)
        for _ in range(2):
            _, r, lam = step(r)
            if t == 0:
                coeffs.append(lam)
        r = _p64(r, eps)
    while len(coeffs) < 4:
        coeffs.append(torch.zeros_like(x[:, :1]))
    c = torch.cat(coeffs, dim=1)

    def closed(a, b):
        outer, inner = a + b, (a - b).abs()
        return torch.stack([-outer, -inner, inner, outer], dim=1)

    cens = [closed(c[:, 0], c[:, 1]), closed(c[:, 2], c[:, 3])]
    if kmeans:
        for f, val in enumerate((u, _p64(x - u - r, eps))):
            cen = cens[f]
            mm = torch.maximum(c[:, 2 * f], c[:, 2 * f + 1])
            bnd = torch.stack([-mm, torch.zeros_like(mm), mm], dim=1)
            for _ in range(kmeans):
                code = sum((val > bnd[:, q:q + 1]).long() for q in range(3))
                cnt = torch.stack([(code == q).sum(1) for q in range(4)], dim=1)
                tot = torch.stack([torch.where(code == q, val, 0.0).sum(1) for q in range(4)], dim=1)
                cen = torch.where(cnt > 0, tot / cnt.clamp(min=1), cen)
                bnd = (cen[:, :3] + cen[:, 1:]) / 2
            cens[f] = cen
    return cens[0], cens[1], c


def _hadamard_block(n):
    return min(n & -n, 16384)


def _hadamard64(x, b):
    m, n = x.shape
    y = x.reshape(-1, b)
    h = 1
    while h < b:
        y = y.reshape(-1, b // (2 * h), 2, h)
        y = torch.stack([y[:, :, 0] + y[:, :, 1], y[:, :, 0] - y[:, :, 1]], dim=2).reshape(-1, b)
        h *= 2
    return (y / math.sqrt(b)).reshape(m, n)


def _plane64(codes, centres, n):
    """Dense float64 rows of one 2-bit plane."""
    shift = 2 * torch.arange(16, device=codes.device)
    q = (codes.long().unsqueeze(2) >> shift & 3).reshape(codes.shape[0], -1)[:, :n]
    return torch.gather(centres.double(), 1, q)


def _rows(m, n):
    """Row ranges of at most 8 M entries."""
    k = max(1, (8 << 20) // n)
    return [slice(a, min(m, a + k)) for a in range(0, m, k)]


def exact(case, seed):
    st = prepare(case, seed)
    op, shapes = case["op"], st["shapes"]
    cols = case.get("layout") == "columns"
    eps = [_signs(s, n) for s, (n, _) in zip(st["seeds"], shapes)]
    out = []
    if op == "quantise":
        for w, e, (n, m) in zip(st["ws"], eps, shapes):
            w = w.t() if cols else w
            got = [_quantise64(w[r], e, case["iters"], case["kmeans"]) for r in _rows(m, n)]
            out.append([None, None] + [torch.cat([g[k] for g in got]) for k in range(3)])
        return out
    if op == "rht":
        for w, e, (n, m) in zip(st["ws"], eps, shapes):
            b = _hadamard_block(n)
            y = torch.empty((m, n), dtype=torch.float64, device="cuda")
            for r in _rows(m, n):
                x = w[r].double()
                y[r] = _hadamard64(x, b) * e if case["inverse"] else _hadamard64(x * e, b)
            out.append(y)
        return out
    if op == "product":
        for x, d, e, (n, m) in zip(st["xs"], st["decs"], eps, shapes):
            x = x.double()
            xp = _p64(x, e)
            y = torch.empty((x.shape[0], m), dtype=torch.float64, device="cuda")
            for r in _rows(m, n):
                y[:, r] = x @ _plane64(d.codes_u[r], d.centres_u[r], n).t() \
                    + xp @ _plane64(d.codes_v[r], d.centres_v[r], n).t()
            out.append(y)
        return out

    def laid(parts):
        y = torch.cat(parts)
        return y.t().contiguous() if cols else y

    us, vs = [], []
    for d, e, (n, m) in zip(st["decs"], eps, shapes):
        u = [_plane64(d.codes_u[r], d.centres_u[r], n) for r in _rows(m, n)]
        v = [_plane64(d.codes_v[r], d.centres_v[r], n) for r in _rows(m, n)]
        if op == "reconstruct":
            out.append(laid([a + _p64(b, e) for a, b in zip(u, v)]))
        else:
            us.append(laid(u))
            vs.append(laid(v))
    return out if op == "reconstruct" else [us, vs]
