"""The work that a user of this library has it do, as cases that can be timed: the data sketch of
dense and sparse tensors, one core update on its own, the relative error, whole sweeps of Algorithm 1
for one tensor and for a batch, and the warm-start network's training pass. Each goes through the
entry points of paper_2309_08093_gb300.lib; sizes are those of the repository's workloads.

listed(): the cases; draw(rng): one more of the same ranges; prepare(case, seed): what a program
holds before the call; run(state): one pass; work(case): the bytes and operations a pass cannot do
without; exact(case, seed): the same outputs in 64 bits from plain torch.

Tensors lie with mode 0 fastest, so a dense tensor is a torch tensor of shape (n[d-1], ..., n[0]) and
a core r0 x n x r1 one of shape (r1, n, r0).
"""
import math
import random

import numpy as np
import torch

from paper_2309_08093_gb300 import lib

LAMBDA = 1e-3       # proximal weight of every workload
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "fp8": 1}
MASK = (1 << 64) - 1


# ---------------------------------------------------------------------------------------------
# the cases

def listed():
    return [
        # the smallest workload (order 3, FP64 storage), a fresh draw per call: latency and launches
        {"name": "sketch-50x50x50-f64", "kind": "sketch", "dims": "50x50x50", "ranks": "1,5,5,1", "J": 1024,
         "dtype": "f64", "fresh": True},
        # the benchmark's tensor, one draw for many tensors (as the warm start's summary takes them)
        {"name": "sketch-100x100x100x100-f32", "kind": "sketch", "dims": "100x100x100x100",
         "ranks": "1,10,10,10,1", "J": 4096, "dtype": "f32", "fresh": False},
        # low-precision storage, order 5, short fibres, the largest J of the workloads
        {"name": "sketch-40x40x40x40x40-fp8", "kind": "sketch", "dims": "40x40x40x40x40",
         "ranks": "1,8,8,8,8,1", "J": 8192, "dtype": "fp8", "fresh": False},
        # odd sizes: fibres that start off the 16-byte grid, a fresh draw per call
        {"name": "sketch-101x84x93x100-bf16", "kind": "sketch", "dims": "101x84x93x100",
         "ranks": "1,10,10,10,1", "J": 1024, "dtype": "bf16", "fresh": True},
        # coordinate form, 20% of the benchmark tensor's entries
        {"name": "sparse-100x100x100x100", "kind": "sparse", "dims": "100x100x100x100",
         "ranks": "1,10,10,10,1", "J": 4096, "nnz": 20000000},
        # a program that drives its own ALS: interface sketch and proximal update of one core
        {"name": "core-100x100x100x100", "kind": "core", "dims": "100x100x100x100", "ranks": "1,10,10,10,1",
         "J": 4096, "k": 1, "fp64": False},
        # the stopping test of an ALS loop
        {"name": "error-100x100x100x100-f32", "kind": "error", "dims": "100x100x100x100",
         "ranks": "1,10,10,10,1", "J": 4096, "dtype": "f32"},
        # a short solve of the smallest workload: ten monitored sweeps in one call
        {"name": "sweep-50x50x50-f64", "kind": "sweep", "dims": "50x50x50", "ranks": "1,5,5,1", "J": 1024,
         "dtype": "f64", "sweeps": 10},
        # the benchmark: monitored sweeps of the order-4 tensor
        {"name": "sweep-100x100x100x100-f32", "kind": "sweep", "dims": "100x100x100x100",
         "ranks": "1,10,10,10,1", "J": 4096, "dtype": "f32", "sweeps": 3},
        # the image-sequence shape of the warm-start family, rank 20 (its last rank at most 3 x 3)
        {"name": "sweep-256x256x3x128-f32", "kind": "sweep", "dims": "256x256x3x128", "ranks": "1,20,3,8,1",
         "J": 2048, "dtype": "f32", "sweeps": 2},
        # a batch of uneven tensors, FP32 and BF16 in turn
        {"name": "batch-32", "kind": "batch", "count": 32, "shapes": 20230919, "sweeps": 1},
        # one pass of the warm-start network's training: loss and gradients of a minibatch
        {"name": "train-256x5144-512-23220", "kind": "train", "batch": 256, "inputs": 5144, "hidden": 512,
         "outputs": 23220},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_shape(rng, orders, n_lo, n_hi, least, most):
    """Mode sizes of a random order whose product lies near a log-uniform total in [least, most]."""
    while True:
        d = rng.choice(orders)
        total = _log_uniform(rng, least, most)
        w = [rng.uniform(0.6, 1.4) for _ in range(d)]
        dims = [int(round(total ** (x / sum(w)))) for x in w]
        if all(n_lo <= n <= n_hi for n in dims) and least / 2 <= math.prod(dims) <= most:
            return dims


def _draw_ranks(rng, dims, lo, hi):
    top = min(hi, min(dims) // 2)
    return [1] + [rng.randint(min(lo, top), top) for _ in dims[1:]] + [1]


def _pow2(x):
    return 1 << max(1, math.ceil(math.log2(x)))


def draw(rng):
    kind = rng.choice(["sketch", "sketch", "sketch", "sparse", "core", "error", "sweep", "sweep", "batch", "train"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(4, 32), "shapes": rng.randrange(1 << 30), "sweeps": 1}
    if kind == "train":
        return {"kind": kind, "batch": rng.randint(32, 256), "inputs": int(_log_uniform(rng, 512, 5144)),
                "hidden": 64 * rng.randint(2, 8), "outputs": int(_log_uniform(rng, 1024, 23220))}
    dims = _draw_shape(rng, [3, 4, 5, 6] if kind == "sketch" else [3, 4, 5], 10, 300, 1e5, 1e8)
    ranks = _draw_ranks(rng, dims, 4, 12)
    smax = max(ranks[k] * ranks[k + 1] for k in range(len(dims)))
    low = _pow2(8 * smax)  # the batched workload's rule, or larger
    c = {"kind": kind, "dims": "x".join(map(str, dims)), "ranks": ",".join(map(str, ranks)),
         "J": min(8192, low << rng.randint(0, 3))}
    if kind == "sparse":
        c["nnz"] = int(_log_uniform(rng, 1e5, min(2e7, math.prod(dims))))
        return c
    if kind == "core":
        c["k"] = rng.randrange(len(dims))
        c["fp64"] = rng.random() < 0.25
        return c
    c["dtype"] = rng.choice(["f64", "f32", "f32", "bf16", "fp8"])
    if kind == "sketch":
        if rng.random() < 0.2:
            c["J"] = rng.choice([150, 200, 1000, 2000])  # the paper's sketch sizes
        c["fresh"] = rng.random() < 0.5
    if kind == "sweep":
        c["sweeps"] = rng.randint(1, 3)
    return c


# ---------------------------------------------------------------------------------------------
# inputs

def _dims(c):
    return [int(x) for x in c["dims"].split("x")]


def _ranks(c):
    return [int(x) for x in c["ranks"].split(",")]


def _rng(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 16 + stream) & ((1 << 62) - 1))
    return g


def _sketch_seed(seed):
    return random.Random(int(seed)).getrandbits(62)


def _true_cores(dims, ranks, seed):
    g = _rng(seed, 1)
    return [torch.randn(ranks[k + 1], n, ranks[k], generator=g, device="cuda") for k, n in enumerate(dims)]


def _start_cores(true, seed):
    """Cores in mid-solve: the tensor's own, each entry off by a tenth of the core's deviation."""
    g = _rng(seed, 2)
    return [t + 0.1 * torch.randn(t.shape, generator=g, device="cuda") for t in true]


def _contract(cores):
    """The dense tensor of TT cores, flat with mode 0 fastest."""
    q = cores[0].reshape(cores[0].shape[0], -1)  # (r1, n0)
    for t in cores[1:]:
        r1, n, r0 = t.shape
        q = (t.reshape(r1 * n, r0) @ q).reshape(r1, -1)
    return q.reshape(-1)


def _store(x, dtype, n0):
    """(storage, scales): FP8 with one scale per mode-0 index, as the library reads it."""
    if dtype == "fp8":
        m = x.reshape(-1, n0)
        scales = (m.abs().amax(0) / 448.0).clamp_min(1e-30)
        return (m / scales).to(torch.float8_e4m3fn).view(torch.uint8).reshape(-1), scales
    return x.to({"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[dtype]), None


def _tensor(true, dtype, seed, noise):
    """Low-rank tensor plus Gaussian noise at a relative Frobenius level, in its storage type."""
    x = _contract(true)
    e = torch.randn(x.numel(), generator=_rng(seed, 3), device="cuda")
    x += (noise * torch.linalg.vector_norm(x) / torch.linalg.vector_norm(e)) * e
    return _store(x, dtype, true[0].shape[1])


def _batch_shapes(c):
    """The batched workload's recipe: order 3-4, modes in [16, 128], ranks in [4, 12], J >= 8 s."""
    r = random.Random(c["shapes"])
    out = []
    for i in range(c["count"]):
        d = r.randint(3, 4)
        dims = [r.randint(16, 128) for _ in range(d)]
        ranks = [1] + [r.randint(4, 12) for _ in range(d - 1)] + [1]
        smax = max(ranks[k] * ranks[k + 1] for k in range(d))
        out.append((dims, ranks, _pow2(8 * smax), "f32" if i % 2 == 0 else "bf16"))
    return out


def _sparse_inputs(c, seed):
    dims, g = _dims(c), _rng(seed, 4)
    idx = torch.stack([torch.randint(0, n, (c["nnz"],), generator=g, device="cuda", dtype=torch.int32) for n in dims])
    return idx, torch.randn(c["nnz"], generator=g, device="cuda")


def _core_inputs(c, seed):
    """Cores with orthonormal outer unfoldings (as inside a sweep) and the sketch of a noisy tensor of
    these cores, Y_k = S H_k G_k^T + noise."""
    dims, ranks, k = _dims(c), _ranks(c), c["k"]
    cores = _right_to_left([_wide(t) for t in _true_cores(dims, ranks, seed)])
    for j in range(k):
        cores[j], cores[j + 1] = _left_step(cores[j], cores[j + 1])
    cores = [_narrow(g) for g in cores]
    hs, vs = _tables(dims, c["J"], _sketch_seed(seed), 0)
    sh = _interface([_wide(t) for t in cores], hs, vs, c["J"], k)
    y = sh @ _wide(cores[k]).permute(2, 0, 1).reshape(-1, dims[k])
    y += 0.01 * y.std() * torch.randn(y.shape, generator=_rng(seed, 5), device="cuda")
    return cores, y.t().contiguous().to(torch.float32)  # (n, J): column i contiguous


def _train_inputs(c, seed):
    """Seeded He-initialised weights, unit inputs and targets."""
    g = _rng(seed, 6)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    i, h, o, b = c["inputs"], c["hidden"], c["outputs"], c["batch"]
    weights = [n(h, i) * math.sqrt(2 / i), 0.01 * n(h), n(h, h) * math.sqrt(2 / h), 0.01 * n(h),
               n(o, h) * math.sqrt(1 / h), 0.01 * n(o)]
    return weights, n(b, i), n(b, o)


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "t": 0}
    if kind == "train":
        weights, s["X"], s["T"] = _train_inputs(c, seed)
        s["mlp"] = lib.Mlp(c["inputs"], c["hidden"], c["outputs"], c["batch"])
        s["mlp"].tt_mlp_set_weights(*weights)
        s["grads"] = [torch.empty_like(w) for w in weights]
        return s
    if kind == "batch":
        s["A"], s["cores"], specs = [], [], []
        for i, (dims, ranks, J, dtype) in enumerate(_batch_shapes(c)):
            true = _true_cores(dims, ranks, seed + 1000 * i)
            s["A"].append(_tensor(true, dtype, seed + 1000 * i, 1e-3)[0])
            s["cores"].append(_start_cores(true, seed + 1000 * i))
            specs.append({"dims": dims, "ranks": ranks, "J": J, "lam": LAMBDA, "dtype": dtype,
                          "seed": _sketch_seed(seed + 1000 * i)})
        s["batch"] = lib.Batch(specs)
        return s
    dims, ranks = _dims(c), _ranks(c)
    flags = lib.TT_FLAG_FP64_SOLVE if c.get("fp64") else 0
    s["ctx"] = lib.Context(dims, ranks, c["J"], LAMBDA, _sketch_seed(seed), c.get("dtype", "f32"), flags)
    if kind == "core":
        s["cores"], s["Y"] = _core_inputs(c, seed)
        s["SH"] = torch.empty(ranks[c["k"]] * ranks[c["k"] + 1], c["J"], device="cuda")
        return s
    if kind in ("sketch", "sparse"):
        s["Y"] = [torch.empty(n, c["J"], device="cuda") for n in dims]
    if kind == "sparse":
        s["idx"], s["val"] = _sparse_inputs(c, seed)
        return s
    true = _true_cores(dims, ranks, seed)
    s["A"], s["scales"] = _tensor(true, c["dtype"], seed, 1e-2)
    if kind != "sketch":
        s["cores"] = _start_cores(true, seed)
    return s


# ---------------------------------------------------------------------------------------------
# one pass

def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "sketch":
        s["ctx"].tt_sketch_unfold(s["A"], -1, s["t"], s["Y"], s["scales"])
        if c["fresh"]:
            s["t"] += 1
        return s["Y"]
    if kind == "sparse":
        s["ctx"].tt_sketch_unfold_coo(s["idx"], s["val"], c["nnz"], -1, 0, s["Y"])
        return s["Y"]
    if kind == "core":
        s["ctx"].tt_sketch_interface(s["cores"], c["k"], 0, s["SH"])
        s["ctx"].tt_prox_update(s["Y"], s["SH"], s["cores"][c["k"]], c["k"])
        return [s["SH"], s["cores"][c["k"]]]
    if kind == "error":
        return s["ctx"].tt_rel_error(s["A"], s["cores"], s["scales"])
    if kind == "sweep":
        err, _ = s["ctx"].tt_prox_als_sweep_monitored(s["A"], s["cores"], c["sweeps"], s["t"], s["scales"])
        s["t"] += c["sweeps"]
        return {"errors": err, "cores": s["cores"]}
    if kind == "batch":
        s["batch"].tt_batch_sweep(s["A"], s["cores"], c["sweeps"], s["t"])
        s["t"] += c["sweeps"]
        return [torch.cat([t.reshape(-1) for t in cores]) for cores in s["cores"]]
    loss = s["mlp"].tt_mlp_loss_grads(s["X"], s["T"], c["batch"], s["grads"])
    return {"loss": loss, "grads": s["grads"]}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without

def _sweep_work(dims, ranks, J, dtype, errors):
    n = math.prod(dims)
    flops, small = len(dims) * n, 0
    for k, nk in enumerate(dims):
        s = ranks[k] * ranks[k + 1]
        small += 8 * s * nk  # the core, read and written
        flops += 2 * J * s * (s + nk) + s ** 3 / 3 + 2 * s * s * nk + 5 * J * math.log2(J) * s
    if errors:
        flops += 2 * n * ranks[1]
    return {"bytes": n * BYTES[dtype] * (2 if errors else 1) + small, "flops": flops}


def work(case):
    c, kind = case, case["kind"]
    if kind == "train":
        i, h, o, b = c["inputs"], c["hidden"], c["outputs"], c["batch"]
        w = i * h + h * h + h * o
        return {"bytes": 8 * w + 4 * b * (i + o), "flops": 2 * b * (3 * w - i * h)}
    if kind == "batch":
        ws = [_sweep_work(d, r, J, t, False) for d, r, J, t in _batch_shapes(c)]
        return {"bytes": c["sweeps"] * sum(w["bytes"] for w in ws), "flops": c["sweeps"] * sum(w["flops"] for w in ws)}
    dims, ranks, J = _dims(c), _ranks(c), c["J"]
    n, d = math.prod(dims), len(dims)
    if kind == "sketch":
        return {"bytes": n * BYTES[c["dtype"]] + 4 * J * sum(dims), "flops": d * n}
    if kind == "sparse":
        return {"bytes": 4 * (d + 1) * c["nnz"] + 4 * J * sum(dims), "flops": d * c["nnz"]}
    if kind == "core":
        k = c["k"]
        s, nk = ranks[k] * ranks[k + 1], dims[k]
        cores = sum(ranks[j] * dims[j] * ranks[j + 1] for j in range(d))
        ffts = 2.5 * J * math.log2(J) * (sum(ranks[j] * ranks[j + 1] for j in range(d) if j != k) + s)
        return {"bytes": 4 * (J * (s + nk) + cores + s * nk), "flops": ffts + 2 * J * s * (s + nk) + s ** 3 / 3 + 2 * s * s * nk}
    if kind == "error":
        return {"bytes": n * BYTES[c["dtype"]], "flops": 2 * n * ranks[1] + 3 * n}
    w = _sweep_work(dims, ranks, J, c["dtype"], True)
    return {"bytes": c["sweeps"] * w["bytes"], "flops": c["sweeps"] * w["flops"]}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits, from the definitions

def _wide(t):
    return t.to(torch.float64).permute(2, 1, 0)  # (r0, n, r1)


def _narrow(g):
    return g.permute(2, 1, 0).contiguous().to(torch.float32)


def _mix(z):
    z = ((z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9))
    z = ((z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB))
    return z ^ (z >> np.uint64(31))


def _tables(dims, J, seed, sweep):
    """The drawn hashes and signs of every mode: chained SplitMix64 steps."""
    step = lambda z, f: _mix(z + (f + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15))  # noqa: E731
    hs, vs = [], []
    with np.errstate(over="ignore"):
        for k, n in enumerate(dims):
            z = step(step(np.array([seed & MASK], dtype=np.uint64), np.uint64(sweep)), np.uint64(k))
            i = np.arange(n, dtype=np.uint64)
            hs.append(torch.from_numpy((step(step(z, np.uint64(0)), i) % np.uint64(J)).astype(np.int64)).cuda())
            neg = (step(step(z, np.uint64(1)), i) >> np.uint64(63)).astype(np.float64)
            vs.append(torch.from_numpy(1.0 - 2.0 * neg).cuda())
    return hs, vs


def _sketch(a, dims, hs, vs, J):
    """Y_k = S A_(k)^T of a dense tensor (flat, FP64) by the definition; each (n_k, J)."""
    d, out = len(dims), []
    view = lambda x, k: x.reshape([-1] + [1] * k)  # noqa: E731  (mode k is axis d - 1 - k)
    bucket = sum(view(h, k) for k, h in enumerate(hs))
    a = a.reshape(dims[::-1]).clone()
    for k, v in enumerate(vs):
        a *= view(v, k)
    for k in range(d):
        at = (bucket - view(hs[k], k)) % J + J * view(torch.arange(dims[k], device="cuda"), k)
        y = torch.zeros(dims[k] * J, dtype=torch.float64, device="cuda")
        y.index_add_(0, at.reshape(-1), (a * view(vs[k], k)).reshape(-1))
        out.append(y.reshape(dims[k], J))
    return out


def _interface(cores, hs, vs, J, k):
    """S H_k as J x s_k, column c = a + r_k b (Theorems 1 and 2)."""
    def spectrum(j):
        g = cores[j] * vs[j][None, :, None]
        x = torch.zeros(g.shape[0], J, g.shape[2], dtype=torch.float64, device="cuda")
        x.index_add_(1, hs[j], g)
        return torch.fft.fft(x, dim=1)

    left = torch.ones(J, 1, dtype=torch.complex128, device="cuda")
    for j in range(k):
        left = torch.einsum("wa,awb->wb", left, spectrum(j))
    right = torch.ones(J, 1, dtype=torch.complex128, device="cuda")
    for j in range(len(cores) - 1, k, -1):
        right = torch.einsum("awb,wb->wa", spectrum(j), right)
    both = torch.einsum("wb,wa->wba", right, left).reshape(J, -1)
    return torch.fft.ifft(both, dim=0).real


def _qr(m):
    """QR with a non-negative diagonal; a wide m gets zero-padded factors."""
    rows, cols = m.shape
    q, r = torch.linalg.qr(m)
    s = torch.where(torch.diagonal(r) < 0, -1.0, 1.0).to(m.dtype)
    q, r = q * s, r * s[:, None]
    if rows < cols:
        q = torch.cat([q, torch.zeros(rows, cols - rows, dtype=m.dtype, device=m.device)], 1)
        r = torch.cat([r, torch.zeros(cols - rows, cols, dtype=m.dtype, device=m.device)], 0)
    return q, r


def _left_step(g, nxt):
    r0, n, r1 = g.shape
    q, r = _qr(g.reshape(r0 * n, r1))
    return q.reshape(r0, n, r1), torch.einsum("ab,bic->aic", r, nxt)


def _right_to_left(cores):
    cores = list(cores)
    for k in range(len(cores) - 1, 0, -1):
        r0, n, r1 = cores[k].shape
        q, r = _qr(cores[k].reshape(r0, n * r1).t())
        cores[k] = q.t().reshape(r0, n, r1)
        cores[k - 1] = torch.einsum("aib,cb->aic", cores[k - 1], r)
    return cores


def _update(y, sh, g):
    """Eq. (ite): y (n, J), sh (J, s), g (r0, n, r1)."""
    r0, n, r1 = g.shape
    g2 = g.permute(1, 2, 0).reshape(n, -1)  # column a + r0 b
    m = sh.t() @ sh + LAMBDA * torch.eye(sh.shape[1], dtype=sh.dtype, device=sh.device)
    x = torch.linalg.solve(m, (y @ sh + LAMBDA * g2).t()).t()
    return x.reshape(n, r1, r0).permute(2, 0, 1)


def _one_sweep(a, dims, cores, J, seed, t):
    hs, vs = _tables(dims, J, seed, t)
    ys = _sketch(a, dims, hs, vs, J)
    cores = _right_to_left(cores)
    for k in range(len(dims)):
        cores[k] = _update(ys[k], _interface(cores, hs, vs, J, k), cores[k])
        if k < len(dims) - 1:
            cores[k], cores[k + 1] = _left_step(cores[k], cores[k + 1])
    return cores


def _error(a, cores):
    x = _contract([g.permute(2, 1, 0) for g in cores])
    return float(torch.linalg.vector_norm(a - x) / torch.linalg.vector_norm(a))


def _decoded(storage, scales, n0):
    if scales is None:
        return storage.to(torch.float64)
    m = storage.view(torch.float8_e4m3fn).to(torch.float64).reshape(-1, n0)
    return (m * scales.to(torch.float64)).reshape(-1)


def _exact_train(c, seed):
    weights, x, t = _train_inputs(c, seed)
    w1, b1, w2, b2, w3, b3 = ws = [w.to(torch.float64).requires_grad_() for w in weights]
    gelu = torch.nn.functional.gelu
    y = gelu(gelu(x.to(torch.float64) @ w1.t() + b1) @ w2.t() + b2) @ w3.t() + b3
    loss = ((y - t.to(torch.float64)) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "grads": [w.grad for w in ws]}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "batch":
        out = []
        for i, (dims, ranks, J, dtype) in enumerate(_batch_shapes(c)):
            si = seed + 1000 * i
            true = _true_cores(dims, ranks, si)
            a = _decoded(*_tensor(true, dtype, si, 1e-3), dims[0])
            cores = [_wide(t) for t in _start_cores(true, si)]
            for t in range(c["sweeps"]):
                cores = _one_sweep(a, dims, cores, J, _sketch_seed(si), t)
            out.append(torch.cat([g.permute(2, 1, 0).reshape(-1) for g in cores]))
        return out
    dims, ranks, J = _dims(c), _ranks(c), c["J"]
    hs, vs = _tables(dims, J, _sketch_seed(seed), 0)
    if kind == "sparse":
        idx, val = _sparse_inputs(c, seed)
        idx = idx.long()
        bucket = sum(h[i] for h, i in zip(hs, idx))
        x = val.to(torch.float64)
        for v, i in zip(vs, idx):
            x = x * v[i]
        out = []
        for k, n in enumerate(dims):
            y = torch.zeros(n * J, dtype=torch.float64, device="cuda")
            y.index_add_(0, (bucket - hs[k][idx[k]]) % J + J * idx[k], x * vs[k][idx[k]])
            out.append(y.reshape(n, J))
        return out
    if kind == "core":
        cores, y = _core_inputs(c, seed)
        wide = [_wide(t) for t in cores]
        sh = _interface(wide, hs, vs, J, c["k"])
        new = _update(y.to(torch.float64), sh, wide[c["k"]])
        return [sh.t().contiguous(), new.permute(2, 1, 0).contiguous()]
    true = _true_cores(dims, ranks, seed)
    a = _decoded(*_tensor(true, c["dtype"], seed, 1e-2), dims[0])
    if kind == "sketch":
        return _sketch(a, dims, hs, vs, J)
    cores = [_wide(t) for t in _start_cores(true, seed)]
    if kind == "error":
        return _error(a, cores)
    errors = []
    for t in range(c["sweeps"]):
        cores = _one_sweep(a, dims, cores, J, _sketch_seed(seed), t)
        errors.append(_error(a, cores))
    return {"errors": errors, "cores": [g.permute(2, 1, 0).contiguous() for g in cores]}
