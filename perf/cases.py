"""The work that a program has this library do, as cases to be timed and compared.

A case is a dict of plain values; `listed()` gives the fixed ones, `draw()` more of the same ranges. Every matrix is
made on the GPU (on the host where the entry point takes host buffers) from the seed alone, with the spectra of the
library's own workloads: exact rank, image-like, slow decay, harmonic, Eq. (mat2), hyperspectral, pixel batch.

Operations:
  factor    one matrix through `factor`: U, D, V                          (compression, rank finding)
  restore   one matrix through `factor` and back through `Factors.reconstruct`: A_hat             (denoising)
  channels  the channels of a colour image through `compress_channels`    (batched entry point, FP64 items)
  batch     many FP32 images of uneven size through `factor_batched`, their factors packed into one buffer each
  host      a host matrix through `factor_host`, factors back on the host
  decode    stored factors back to a matrix through `eod_abe_reconstruct`

Where the tolerance and not the matrix decides the rank, the factors are stored in buffers of `cap` columns, zero
beyond the rank (as `factor_host` fills them). FP32 and mixed factorisations are run where their factors are
determined to FP32's own accuracy (a relative tolerance of 0.02 and more: the paper's images stop at 0.036) or
return what U, D and V give together. Their D is stored with U and V in the factors' type, as a program that writes
them to one file does.
"""
import ctypes
import math

import torch

import paper_2506_22713_gb300 as eod

F64, F32 = torch.float64, torch.float32
TYPES = {"f64": F64, "f32": F32}


def listed():
    return [
        # The smallest call: a 512 x 384 matrix of exact rank 20 (the rank-revealing setting of Thm 3.4); one block,
        # where launches, host round trips and the small factorisations are all there is.
        {"name": "exact_512x384_f64", "op": "factor", "kind": "exact", "m": 512, "n": 384, "r": 20, "dtype": "f64",
         "precision": "plain", "tol": 1e-10, "mode": "abs", "tau": 0},
        # The colour image of Sec. 1: three 220 x 220 channels of ranks near 50, compressed in one call.
        {"name": "rgb_220_f64", "op": "channels", "kind": "nonneg", "m": 220, "n": 220, "r": 50, "count": 3,
         "dtype": "f64", "precision": "plain", "tol": 1e-10, "mode": "rel", "tau": 0},
        # The robustness suite's size (Matrix IV of Sec. 4.3, n = 1000): a mid-size FP64 matrix of rank about 105.
        {"name": "slow_1000_f64", "op": "factor", "kind": "slow", "m": 1000, "n": 1000, "r": 105, "cap": 160, "dtype": "f64",
         "precision": "plain", "tol": 1e-3, "mode": "rel", "tau": 0},
        # The same from host memory and back, of odd, uneven size: what a program without device buffers calls.
        {"name": "host_1501x1103_f64", "op": "host", "kind": "slow", "m": 1501, "n": 1103, "r": 35, "dtype": "f64",
         "precision": "plain", "tol": 5e-3, "mode": "rel", "tau": 0},
        # The image-like matrix of the benchmark, of nearly full rank at its tolerance: the method's worst case.
        {"name": "image_2048_f64", "op": "factor", "kind": "image", "m": 2048, "n": 2048, "r": 2037, "cap": 2048, "dtype": "f64",
         "precision": "plain", "tol": 1e-3, "mode": "rel", "tau": 0},
        # Eq. (mat2) at the first size of the paper's timing table, with one subspace iteration.
        {"name": "mat2_4000_tau1_f64", "op": "factor", "kind": "uniform", "m": 4000, "n": 4000, "r": 1600,
         "dtype": "f64", "precision": "plain", "tol": 1e-8, "mode": "abs", "tau": 1},
        # The hyperspectral cube, unfolded: a very tall FP32 matrix of rank 13, bound by passes over the data.
        {"name": "hyper_262144x224_mixed", "op": "factor", "kind": "hyper", "m": 262144, "n": 224, "r": 13, "cap": 32,
         "dtype": "f32", "precision": "mixed", "tol": 0.047, "mode": "rel", "tau": 0},
        # The benchmark's headline: the 8192 x 8192 harmonic matrix in the mixed BF16 form, and A_hat from its factors.
        {"name": "harmonic_8192_mixed", "op": "restore", "kind": "harmonic", "m": 8192, "n": 8192, "r": 455,
         "dtype": "f32", "precision": "mixed", "tol": 0.0128, "mode": "rel", "tau": 0},
        # An odd-sized FP32 matrix of a few thousand in the mixed TF32 form, and one in plain FP32.
        {"name": "harmonic_3001x2503_tf32", "op": "restore", "kind": "harmonic", "m": 3001, "n": 2503, "r": 313,
         "dtype": "f32", "precision": "mixed_tf32", "tol": 0.03, "mode": "rel", "tau": 0},
        {"name": "harmonic_1537x2049_f32", "op": "factor", "kind": "harmonic", "m": 1537, "n": 2049, "r": 326, "cap": 400,
         "dtype": "f32", "precision": "plain", "tol": 0.03, "mode": "rel", "tau": 0},
        # The batch of 256 images of uneven size, in the one persistent launch.
        {"name": "batch_256_f32", "op": "batch", "kind": "pixels", "m": 2048, "n": 2048, "r": 128, "count": 256,
         "dtype": "f32", "precision": "plain", "tol": 0.02, "mode": "rel", "tau": 0},
        # Decoding a stored image: A_hat = U D V^T in FP64.
        {"name": "decode_2048_f64", "op": "decode", "kind": "stored", "m": 2048, "n": 2048, "r": 600, "dtype": "f64",
         "precision": "plain", "tol": 0.0, "mode": "rel", "tau": 0},
    ]


def draw(rng):
    """One more case: the same operations and spectra, sizes over the whole range (odd ones among them)."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def tol(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    pick = rng.choice(["exact", "channels", "slow", "host", "image", "uniform", "hyper", "harmonic", "batch", "decode"])
    c = {"op": "factor", "kind": pick, "dtype": "f64", "precision": "plain", "mode": "rel", "tau": 0}
    if pick == "exact":
        m, n = size(256, 2048), size(256, 2048)
        c.update(m=m, n=n, r=rng.randint(5, 60), tol=1e-10, mode="abs")
    elif pick == "channels":
        c.update(op="channels", kind="nonneg", m=size(160, 640), n=size(160, 640), r=rng.randint(20, 60), count=3, tol=1e-10)
    elif pick in ("slow", "host"):
        c.update(op="factor" if pick == "slow" else "host", kind="slow", m=size(600, 2200), n=size(600, 2200), tol=tol(1e-3, 1e-2))
        c["r"] = int(0.85 * c["tol"] ** -0.7)
        c["cap"] = min(c["m"], c["n"], 2 * c["r"] + 32)
    elif pick == "image":
        c.update(m=size(512, 2048), n=size(512, 2048), tol=1e-3)
        c["r"], c["cap"] = int(0.99 * min(c["m"], c["n"])), min(c["m"], c["n"])
    elif pick == "uniform":
        n = size(1000, 4000)
        c.update(m=n, n=n, r=int(0.4 * n), tol=1e-8, mode="abs", tau=rng.choice([0, 1]))
    elif pick == "hyper":
        c.update(m=size(30000, 262144), n=rng.randint(150, 260), r=13, cap=32, dtype="f32", tol=0.047,
                 precision=rng.choice(["mixed", "mixed", "mixed_tf32", "plain"]))
    elif pick == "harmonic":
        c.update(op="restore", m=size(1200, 8192), n=size(1200, 8192), dtype="f32", tol=tol(0.0128, 0.05),
                 precision=rng.choice(["mixed", "mixed_tf32", "plain"]))
        c["r"] = min(int(9.0 / c["tol"]), 450)
    elif pick == "batch":
        c.update(op="batch", kind="pixels", m=size(512, 2048), n=size(512, 2048), r=128, count=size(32, 256), dtype="f32", tol=0.02)
    else:
        dt = rng.choice(["f64", "f32"])
        c.update(op="decode", kind="stored", dtype=dt, m=size(256, 4096 if dt == "f32" else 2048),
                 n=size(256, 4096 if dt == "f32" else 2048), tol=0.0)
        c["r"] = max(8, int(min(c["m"], c["n"]) * rng.uniform(0.05, 0.4)))
    return c


# --------------------------------------------------------------------------------------------------------- inputs --

def _frame(g, m, r):
    """m x r, orthonormal columns: the Q of a Gaussian."""
    return torch.linalg.qr(torch.randn(m, r, generator=g, device="cuda", dtype=F64))[0]


def _product(L, s, R, dtype, noise=0.0, g=None):
    """L diag(s) R^T (+ noise), column-major."""
    At = (R * s) @ L.t()
    if noise:
        At += noise * torch.randn(At.shape, generator=g, device="cuda", dtype=F64)
    return At.to(dtype).t()


def _index(r):
    return torch.arange(1, r + 1, device="cuda", dtype=F64)


def _uneven(case):
    """The sizes and ranks of a batch's items: rows and columns over [256, the case's], ranks over [8, 128]."""
    g = torch.Generator().manual_seed(case["m"] * 4099 + case["n"])
    u = torch.rand(case["count"], 3, generator=g, dtype=F64)
    return [(256 + int(a * (case["m"] - 255)), 256 + int(b * (case["n"] - 255)), 8 + int(c * (case["r"] - 7))) for a, b, c in u.tolist()]


def _matrices(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, n, r, kind, dt = case["m"], case["n"], case["r"], case["kind"], TYPES[case["dtype"]]
    if kind == "exact":      # singular values geometric from 1 to 1e-2, nothing else
        return [_product(_frame(g, m, r), 10.0 ** (-2.0 * (_index(r) - 1) / max(r - 1, 1)), _frame(g, n, r), dt)]
    if kind == "nonneg":     # products of non-negative factors, scaled to [0, 255]
        out = []
        for i in range(case["count"]):
            C = torch.rand(n, r + i, generator=g, device="cuda", dtype=F64) @ torch.rand(r + i, m, generator=g, device="cuda", dtype=F64)
            out.append((C * (255.0 / C.max())).to(dt).t())
        return out
    if kind == "slow":       # sigma_i = i^-2
        q = min(m, n)
        return [_product(_frame(g, m, q), _index(q) ** -2.0, _frame(g, n, q), dt)]
    if kind == "image":      # sigma_i = 255 i^-1.5 (150 of them) over noise of 1e-4 of the largest
        q = min(150, m, n)
        return [_product(_frame(g, m, q), 255.0 * _index(q) ** -1.5, _frame(g, n, q), dt, 1e-4 * 255.0, g)]
    if kind == "uniform":    # Eq. (mat2): r values uniform in (0, 1), sorted
        s = torch.rand(r, generator=g, device="cuda", dtype=F64).sort(descending=True).values
        return [_product(_frame(g, m, r), s, _frame(g, n, r), dt)]
    if kind == "harmonic":   # sigma_i = 1/i (400 of them) over noise of 1e-6
        q = min(400, m, n)
        return [_product(_frame(g, m, q), 1.0 / _index(q), _frame(g, n, q), dt, 1e-6, g)]
    if kind == "hyper":      # Dirichlet abundances x smooth spectra of 12 endmembers, 30 dB noise
        W = -torch.log(torch.rand(12, m, generator=g, device="cuda", dtype=F64).clamp_min(1e-300))
        W = W / W.sum(0)
        p = torch.rand(3, 12, 5, generator=g, device="cuda", dtype=F64)
        at = torch.arange(n, device="cuda", dtype=F64)
        S = ((0.1 + 0.9 * p[0]).unsqueeze(2) * torch.exp(-((at - n * p[1].unsqueeze(2)) ** 2) / (2.0 * (4.0 + 36.0 * p[2].unsqueeze(2)) ** 2))).sum(1)
        X = S.t() @ W
        return [(X + X.norm() / math.sqrt(X.numel() * 1e3) * torch.randn(n, m, generator=g, device="cuda", dtype=F64)).to(dt).t()]
    assert kind == "pixels"  # sigma_i = 255 exp(-4 i / r), near-orthonormal Gaussian factors, uneven sizes
    out = []
    for mi, ni, ri in _uneven(case):
        L = torch.randn(mi, ri, generator=g, device="cuda", dtype=F64) / math.sqrt(mi)
        R = torch.randn(ni, ri, generator=g, device="cuda", dtype=F64) / math.sqrt(ni)
        out.append(_product(L, 255.0 * torch.exp(-4.0 * _index(ri) / ri), R, dt))
    return out


def _stored(case, seed):
    """Factors as a program reads them back: U, V with orthonormal columns, D upper triangular with a decaying diagonal."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, n, r, dt = case["m"], case["n"], case["r"], TYPES[case["dtype"]]
    D = torch.randn(r, r, generator=g, device="cuda", dtype=F64).triu(1) / math.sqrt(r) + torch.diag(1.0 + torch.rand(r, generator=g, device="cuda", dtype=F64))
    D = D * (255.0 * _index(r) ** -1.0).unsqueeze(1)
    return _frame(g, m, r).to(dt).t().contiguous().t(), D.t().contiguous().t(), _frame(g, n, r).to(dt).t().contiguous().t()


def _omega_seed(seed):
    return seed * 7919 + 11


def prepare(case, seed):
    s = dict(case, seed=_omega_seed(seed))
    if case["op"] == "decode":
        s["U"], s["D"], s["V"] = _stored(case, seed)
        f = eod.EodFactors(m=case["m"], n=case["n"], rank=case["r"], precision=eod.EOD_PLAIN,
                           f_dtype=eod.EOD_F64 if case["dtype"] == "f64" else eod.EOD_F32)
        f.U, f.D, f.V = s["U"].data_ptr(), s["D"].data_ptr(), s["V"].data_ptr()
        s["f"] = f
        return s
    s["A"] = _matrices(case, seed)
    if case["op"] == "host":
        def pinned(rows, cols):
            return torch.zeros(cols, rows, dtype=F64).pin_memory().t()
        m, n, q = case["m"], case["n"], min(case["m"], case["n"])
        s["A"] = [s["A"][0].t().cpu().pin_memory().t()]
        s["U"], s["D"], s["V"] = pinned(m, q), pinned(q, q), pinned(n, q)
    return s


# ----------------------------------------------------------------------------------------------------------- calls --

def _columns(X, cap):
    """X in a buffer of cap columns, zero beyond its own."""
    return torch.nn.functional.pad(X.t(), (0, 0, 0, cap - X.shape[1])).t()


def _kept(rank, U, D, V, cap=None):
    if cap is not None:
        U, D, V = _columns(U, cap), torch.nn.functional.pad(D.t(), (0, cap - rank, 0, cap - rank)).t(), _columns(V, cap)
    return {"rank": rank, "U": U, "D": D, "V": V}


def _factors(f, cap=None):
    return _kept(f.rank, f.U, f.D.to(f.f_dtype), f.V, cap)


def _packed(case, ranks, U, D, V):
    """The factors of a batch one after another in one buffer for each of U, D and V, zero beyond the last."""
    def pack(ts, most):
        used = sum(t.numel() for t in ts)
        return torch.cat([t.t().reshape(-1) for t in ts] + [ts[0].new_zeros(most - used)])
    most = [min(i) for i in _uneven(case)]
    return {"rank": torch.tensor(ranks), "U": pack(U, sum(i[0] * q for i, q in zip(_uneven(case), most))),
            "D": pack(D, sum(q * q for q in most)), "V": pack(V, sum(i[1] * q for i, q in zip(_uneven(case), most)))}


def run(s):
    how = {"precision": s["precision"], "tol_mode": s["mode"], "power_iters": s["tau"]}
    if s["op"] == "factor":
        return _factors(eod.factor(s["A"][0], s["tol"], s["seed"], **how), s.get("cap"))
    if s["op"] == "restore":
        f = eod.factor(s["A"][0], s["tol"], s["seed"], **how)
        return {"rank": f.rank, "A_hat": f.reconstruct()}
    if s["op"] == "channels":
        report, fs = eod.compress_channels(s["A"], s["tol"], s["seed"], **how)
        return [_factors(f) for f in fs]
    if s["op"] == "batch":
        fs = eod.factor_batched(s["A"], s["tol"], s["seed"], **how)[0]
        p = _packed(s, [f.rank for f in fs], [f.U for f in fs], [f.D for f in fs], [f.V for f in fs])
        return dict(p, D=p["D"].to(fs[0].f_dtype))
    if s["op"] == "host":
        rank, err = eod.factor_host(s["A"][0], s["tol"], s["seed"], U_out=s["U"], D_out=s["D"], V_out=s["V"], **how)
        return {"rank": rank, "U": s["U"], "D": s["D"], "V": s["V"]}
    out = torch.empty(s["n"], s["m"], dtype=TYPES[s["dtype"]], device="cuda").t()
    o = eod.make_opts(dtype=s["f"].f_dtype)
    status = eod.eod_abe_reconstruct(ctypes.byref(s["f"]), ctypes.c_void_p(out.data_ptr()), s["m"], ctypes.byref(o))
    if status != eod.EOD_OK:
        raise eod.EodError(status, "eod_abe_reconstruct")
    return out


def work(case):
    """The matrix in and the factors out once each; the products of the paper's cost model (Sec. 3.4) without the
    blocks' share, with the error's, and 4mnr multiply-adds for each subspace iteration."""
    size = 8 if case["dtype"] == "f64" else 4
    if case["op"] == "decode":
        m, n, r = case["m"], case["n"], case["r"]
        return {"bytes": size * (m * r + n * r + m * n) + 8 * r * r, "flops": m * r * r + 2 * m * n * r}
    items = _uneven(case) if case["op"] == "batch" else [(case["m"], case["n"], case["r"])] * case.get("count", 1)
    b = f = 0
    for m, n, r in items:
        b += size * (m * n + m * r + n * r) + 8 * r * r
        f += 2 * (2 * m * n * r + m * r * r + 2 * n * r * r + 2 * r * r * r) + 2 * m * n * r + case["tau"] * 4 * m * n * r
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------------------------- in 64 bits, plain --

def _omega(n, cols, seed, batch):
    """The Gaussian test matrix: Philox4x32-10 on (row, column, batch, 0), Box-Muller, rounded to 8 significant bits."""
    mask = 0xFFFFFFFF
    c = [torch.arange(n, device="cuda").unsqueeze(1).expand(n, cols), torch.arange(cols, device="cuda").expand(n, cols),
         torch.full((n, cols), batch, device="cuda"), torch.zeros(n, cols, dtype=torch.int64, device="cuda")]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # the low 64 bits: all of a product of two 32-bit words
        c = [((b >> 32) & mask) ^ c[1] ^ k0, b & mask, ((a >> 32) & mask) ^ c[3] ^ k1, a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u1, u2 = (c[0].to(F64) + 0.5) * 2.0 ** -32, (c[1].to(F64) + 0.5) * 2.0 ** -32
    frac, exp = torch.frexp(torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2))
    return torch.ldexp(torch.round(frac * 256.0) / 256.0, exp)


def _qr(X):
    """Q and R with a non-negative diagonal."""
    Q, R = torch.linalg.qr(X)
    s = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(F64)
    return Q * s, R * s.unsqueeze(1)


def _decomposed(A, case, seed, batch):
    A = A.to(F64)
    m, n = A.shape
    eps = case["tol"] * (float(A.norm()) if case["mode"] == "rel" else 1.0)
    cols = min(m, n, case["r"] + 64)
    while True:
        Q, R = _qr(A @ _omega(n, cols, seed, batch))
        small = (torch.diagonal(R) <= eps).nonzero()
        if len(small) or cols == min(m, n):
            break
        cols = min(m, n, 2 * cols)
    Q = Q[:, :int(small[0]) if len(small) else cols]
    for _ in range(case["tau"]):
        Q = _qr(A @ _qr(A.t() @ Q)[0])[0]
    V, R = _qr(A.t() @ Q)
    Qh, D = _qr(R.t())
    return {"rank": Q.shape[1], "U": Q @ Qh, "D": D, "V": V}


def exact(case, seed):
    if case["op"] == "decode":
        U, D, V = _stored(case, seed)
        return U.to(F64) @ D @ V.to(F64).t()
    every = [_decomposed(A, case, _omega_seed(seed), i) for i, A in enumerate(_matrices(case, seed))]
    if case["op"] == "channels":
        return every
    if case["op"] == "batch":
        return _packed(case, [d["rank"] for d in every], *([d[k] for d in every] for k in ("U", "D", "V")))
    d = every[0]
    if case["op"] == "restore":
        return {"rank": d["rank"], "A_hat": d["U"] @ d["D"] @ d["V"].t()}
    return _kept(d["rank"], d["U"], d["D"], d["V"], min(case["m"], case["n"]) if case["op"] == "host" else case.get("cap"))
