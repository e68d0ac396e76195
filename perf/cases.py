"""The work this library is used for, as cases that can be timed and compared.

Every case goes through the public bindings (``nla``, ``kt``) as a user's program does: the
shipped table of tuned configurations is installed, workspaces are made once and kept, inputs
are preserved so that the same matrix can be used again.

Kinds of case

* ``svd``   -- singular values of one dense matrix (``nla.gesvd_vals``), FP32 or FP64; for FP64
  matrices also the TF32 / BF16 trailing update and its compensated forms.
* ``batch`` -- singular values of many uneven FP32 matrices in one call
  (``nla.gesvd_vals_batched``).
* ``band``  -- the stages on their own: an upper band matrix to bidiagonal form
  (``nla.band2bd``) and its singular values (``nla.bdsvd_vals``).
* ``mlp``   -- one training step of the tuner's cost model (forward, backward, Adam).
"""
import math
import os

import numpy as np
import torch

from paper_2608_21227_gb300 import inputs, kt, nla

TABLE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_21227_gb300", "tuned",
                     "gb300.kt")
DEFAULT_CFG = (32, 64, 128, 2, 1)  # the fixed default configuration (band 32, tile 64)
UPDATES = {"native": nla.UPD_NATIVE, "tf32": nla.UPD_TF32, "bf16": nla.UPD_BF16, "tf32x3": nla.UPD_TF32X3,
           "bf16x3": nla.UPD_BF16X3}
TYPES = {"f32": torch.float32, "f64": torch.float64}
# exact() answers where the reference in 64 bits takes no more than some seconds
EXACT_MAX_MN2 = 6.0e11
EXACT_BATCH_FLOPS = 2.0e10


def _svd(name, m, n, dtype, values, update="native", default_cfg=False):
    return {"name": name, "kind": "svd", "m": m, "n": n, "dtype": dtype, "values": values, "update": update,
            "default_cfg": default_cfg}


def listed():
    return [
        # a single small call: a 96 x 64 block inside a larger program, all launch latency
        _svd("svd_f32_96x64", 96, 64, "f32", "normal"),
        # the plain method as it is first tried: 256 x 256 FP64, the fixed default configuration
        _svd("svd_f64_256_default", 256, 256, "f64", "normal", default_cfg=True),
        # a wide, ragged matrix (fewer rows than columns: it is transposed into the workspace)
        _svd("svd_f32_650x1001", 650, 1001, "f32", "normal"),
        # the smallest size that the tuner sweeps
        _svd("svd_f32_1024", 1024, 1024, "f32", "uniform"),
        # a tall matrix with odd sizes
        _svd("svd_f32_3001x1537", 3001, 1537, "f32", "uniform"),
        # the benchmark's headline: 8192 x 8192 FP32
        _svd("svd_f32_8192", 8192, 8192, "f32", "uniform"),
        # the FP64 path at a middle size of the tuner's sweep
        _svd("svd_f64_2048", 2048, 2048, "f64", "uniform"),
        # mixed precision: the 4:1 tall shape of that workload, geometric singular values
        _svd("svd_tf32_4096x1024", 4096, 1024, "f64", "geometric", update="tf32"),
        # the batched workload of the benchmark: 10,000 uneven matrices, n in 8..256, m/n in 1..4
        {"name": "batch_10000", "kind": "batch", "count": 10000, "n_lo": 8, "n_hi": 256, "shapes": 3},
        # a small batch of small matrices (a layer's worth of blocks, say)
        {"name": "batch_300_small", "kind": "batch", "count": 300, "n_lo": 8, "n_hi": 64, "shapes": 33},
        # the stages on their own: a band matrix that the caller already has
        {"name": "band_f32_3000_b32", "kind": "band", "n": 3000, "b": 32, "dtype": "f32"},
        # one step of the cost model's training on a large batch of measurements
        {"name": "mlp_step_4096", "kind": "mlp", "rows": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["f32", "f64", "mixed", "batch", "band", "mlp"], weights=[8, 4, 3, 5, 2, 1])[0]
    if kind in ("f32", "f64", "mixed"):
        # any size, square to 4:1, either way up; FP64 work is kept below the largest listed case's time
        n = _log_int(rng, *{"f32": (32, 6000), "f64": (32, 2048), "mixed": (256, 1500)}[kind])
        m = int(n * (1.0 if rng.random() < 0.4 else rng.uniform(1.0, 4.0)))
        m = min(m, 8192 if kind == "f32" else 4096)
        if rng.random() < 0.3:
            m, n = n, m
        small = min(m, n) <= 1024
        values = rng.choice(["normal", "uniform", "geometric"] if small else ["normal", "uniform"])
        update = rng.choice(["tf32", "bf16", "tf32x3", "bf16x3"]) if kind == "mixed" else "native"
        c = _svd("", m, n, "f32" if kind == "f32" else "f64", values, update)
    elif kind == "batch":
        lo = rng.choice([2, 8, 24])
        c = {"name": "", "kind": "batch", "count": _log_int(rng, 40, 9000), "n_lo": lo,
             "n_hi": _log_int(rng, 32, 256), "shapes": rng.randrange(1 << 20)}
    elif kind == "band":
        c = {"name": "", "kind": "band", "n": _log_int(rng, 128, 4000), "b": rng.choice([8, 16, 32, 64]),
             "dtype": rng.choice(["f32", "f32", "f64"])}
        if c["dtype"] == "f64":
            c["n"] = min(c["n"], 1500)
    else:
        c = {"name": "", "kind": "mlp", "rows": _log_int(rng, 200, 16000)}
    del c["name"]
    return c


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _haar(rows, p, g):
    """rows x p with orthonormal columns (QR of a Gaussian matrix, sign fixed)."""
    q, r = torch.linalg.qr(torch.randn(rows, p, generator=g, device="cuda", dtype=torch.float64))
    s = torch.sign(torch.diagonal(r))
    s[s == 0] = 1.0
    return q * s


def _matrix(case, seed):
    """The column-major m x n matrix as a row-major (n, m) tensor."""
    m, n, g = case["m"], case["n"], _generator(seed)
    if case["values"] == "normal":
        a = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64)
    elif case["values"] == "uniform":
        a = torch.rand(n, m, generator=g, device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0)
    else:  # geometric singular values 1 .. 1e-4 between random orthogonal factors
        p = min(m, n)
        sigma = torch.from_numpy(inputs.geometric_sigma(p, 1e4)).cuda()
        a = (_haar(n, p, g) * sigma) @ _haar(m, p, g).T
    return a.to(TYPES[case["dtype"]]).contiguous()


def _batch(case, seed):
    """The matrices of a batch as views of one buffer (row-major (n, m), that is column-major m x n)."""
    ms, ns = inputs.batch_shapes(case["count"], case["shapes"], case["n_lo"], max(case["n_lo"], case["n_hi"]))
    sizes = [int(m) * int(n) for m, n in zip(ms, ns)]
    flat = torch.randn(sum(sizes), generator=_generator(seed), device="cuda", dtype=torch.float32)
    return [a.view(int(n), int(m)) for a, m, n in zip(flat.split(sizes), ms, ns)]


def _band(case, seed):
    """Compact storage (n, 3b+1) of an upper band matrix: entry (i, j) at [j, 2b + i - j]."""
    n, b = case["n"], case["b"]
    ab = torch.zeros(n, 3 * b + 1, device="cuda", dtype=torch.float64)
    ab[:, b:2 * b + 1] = torch.randn(n, b + 1, generator=_generator(seed), device="cuda", dtype=torch.float64)
    j = torch.arange(n, device="cuda")[:, None]
    q = torch.arange(3 * b + 1, device="cuda")[None, :]
    ab[(j + q - 2 * b) < 0] = 0.0
    return ab.to(TYPES[case["dtype"]])


def _mlp(case, seed):
    """Parameters, features and targets, and Adam's moments as some steps of training leave them."""
    g = _generator(seed)
    dims = (kt.FEATURES, 128, 128, 128, 1)
    parts = []
    for i, o in zip(dims[:-1], dims[1:]):
        lim = math.sqrt(6.0 / i)
        parts += [(torch.rand(i * o, generator=g, device="cuda") * 2 - 1) * lim,
                  torch.rand(o, generator=g, device="cuda") * 0.02 - 0.01]
    params = torch.cat(parts)
    X = torch.randn(case["rows"], kt.FEATURES, generator=g, device="cuda")
    y = torch.randn(case["rows"], generator=g, device="cuda")
    m = torch.randn(params.numel(), generator=g, device="cuda") * 0.01
    v = torch.rand(params.numel(), generator=g, device="cuda") * 0.01 + 0.01
    return params, X, y, m, v


MLP_LR, MLP_T = 1e-3, 20


def prepare(case, seed):
    kt.load_config(TABLE)
    s = {"kind": case["kind"]}
    if case["kind"] == "svd":
        a = _matrix(case, seed)
        cfg = nla.Cfg.make(*DEFAULT_CFG) if case["default_cfg"] else None
        upd, p = UPDATES[case["update"]], min(case["m"], case["n"])
        code = nla.F32 if case["dtype"] == "f32" else nla.F64
        need = nla.gesvd_vals_workspace(case["m"], case["n"], code, update=upd, cfg=cfg, preserve_a=True)
        s.update(a=a, cfg=cfg, update=upd, work=nla.workspace(need),
                 S=torch.empty(p, dtype=a.dtype, device="cuda"),
                 info=torch.zeros(1, dtype=torch.int32, device="cuda"))
    elif case["kind"] == "batch":
        b = nla.Batch(_batch(case, seed))
        # the values of all matrices side by side in one buffer
        sizes = [x.numel() for x in b.S]
        s["values"] = torch.empty(sum(sizes), dtype=torch.float32, device="cuda")
        b.S = list(s["values"].split(sizes))
        b.sptrs = torch.tensor([x.data_ptr() for x in b.S], dtype=torch.int64, device="cuda")
        s["batch"] = b
    elif case["kind"] == "band":
        s.update(ab=_band(case, seed), b=case["b"], dtype=TYPES[case["dtype"]])
    else:
        s["params"], s["X"], s["y"], s["m"], s["v"] = _mlp(case, seed)
    return s


def run(s):
    if s["kind"] == "svd":
        S, info = nla.gesvd_vals(s["a"], update=s["update"], cfg=s["cfg"], preserve_a=True, work=s["work"], S=s["S"],
                                 info=s["info"])
        return {"S": S, "info": info}
    if s["kind"] == "batch":
        _, info = nla.gesvd_vals_batched(s["batch"])
        return {"S": s["values"], "info": info}
    if s["kind"] == "band":
        # (d, e) go straight on: the signs and the fine digits of a bidiagonal are not determined by the matrix
        d, e, info = nla.band2bd(s["ab"].clone(), s["b"])  # the chase works in place
        S, info2 = nla.bdsvd_vals(d, e, dtype=s["dtype"])
        return {"S": S, "info": info, "info2": info2}
    pred, grads = kt.mlp_forward_backward(s["params"], s["X"], s["y"])
    kt.mlp_adam_step(s["params"], grads, s["m"], s["v"], MLP_T, MLP_LR)
    return {"pred": pred, "grads": grads, "params": s["params"], "m": s["m"], "v": s["v"]}


def _svd_flops(m, n):
    p, q = float(max(m, n)), float(min(m, n))
    return 4.0 * p * q * q - 4.0 / 3.0 * q ** 3


def work(case):
    if case["kind"] == "svd":
        m, n, e = case["m"], case["n"], 4 if case["dtype"] == "f32" else 8
        return {"bytes": e * (m * n + min(m, n)), "flops": _svd_flops(m, n)}
    if case["kind"] == "batch":
        ms, ns = inputs.batch_shapes(case["count"], case["shapes"], case["n_lo"], max(case["n_lo"], case["n_hi"]))
        return {"bytes": 4.0 * float(np.sum(ms * ns + ns)), "flops": float(sum(_svd_flops(m, n) for m, n in zip(ms, ns)))}
    if case["kind"] == "band":
        n, b, e = case["n"], case["b"], 4 if case["dtype"] == "f32" else 8
        return {"bytes": float(e * n * (b + 2)), "flops": 8.0 * b * n * n}
    rows, par = case["rows"], kt.mlp_param_count()
    return {"bytes": 4.0 * (rows * (kt.FEATURES + 2) + 7 * par), "flops": 6.0 * rows * par}


def exact(case, seed):
    if case["kind"] == "svd":
        p, q = max(case["m"], case["n"]), min(case["m"], case["n"])
        if float(p) * q * q > EXACT_MAX_MN2:
            return None
        return {"S": torch.linalg.svdvals(_matrix(case, seed).double(), driver="gesvd"), "info": None}
    if case["kind"] == "batch":
        if work(case)["flops"] > EXACT_BATCH_FLOPS:
            return None
        return {"S": np.concatenate([np.linalg.svd(a.double().cpu().numpy(), compute_uv=False)
                                     for a in _batch(case, seed)]), "info": None}
    if case["kind"] == "band":
        n, b = case["n"], case["b"]
        if float(n) ** 3 > EXACT_MAX_MN2:
            return None
        ab = _band(case, seed).double()
        a = torch.zeros(n, n, device="cuda", dtype=torch.float64)
        for k in range(min(b, n - 1) + 1):  # the k-th superdiagonal
            a.diagonal(k).copy_(ab[k:, 2 * b - k])
        return {"S": torch.linalg.svdvals(a, driver="gesvd"), "info": None, "info2": None}
    params, X, y, m, v = (t.double() for t in _mlp(case, seed))
    dims, layers, at = (kt.FEATURES, 128, 128, 128, 1), [], 0
    params.requires_grad_(True)
    for i, o in zip(dims[:-1], dims[1:]):
        layers.append((params[at:at + i * o].view(o, i), params[at + i * o:at + i * o + o]))
        at += i * o + o
    h = X
    for k, (W, c) in enumerate(layers):
        h = h @ W.T + c
        h = torch.relu(h) if k < 3 else h
    pred = h[:, 0]
    grads, = torch.autograd.grad(((pred - y) ** 2).mean(), params)
    m = 0.9 * m + 0.1 * grads
    v = 0.999 * v + 0.001 * grads * grads
    new = params - MLP_LR * (m / (1 - 0.9 ** MLP_T)) / (torch.sqrt(v / (1 - 0.999 ** MLP_T)) + 1e-8)
    return {"pred": pred.detach(), "grads": grads, "params": new.detach(), "m": m, "v": v}
