"""The cases libtsqr's speed is measured on: what its callers do with it, through the public calls
of the ``paper_1002_4250_gb300`` package, from a 10,000 x 16 matrix to gigabytes.

A matrix is column-major, held by an (n, lda) tensor.  Entries are iid N(0, 1), or, with
``kappa``, G diag(sigma) V^T with N(0, 1) G, orthogonal V and singular values spaced
geometrically from 1 to 1/kappa (the columns of a regression matrix are never independent).
Sizes are those of this repository's benchmark and tests, and odd ones between them.
"""
import math

import torch

import paper_1002_4250_gb300 as tsqr

_DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # the smallest matrix worth a GPU: a caller waits for launches and dependent steps
        {"name": "r f64 10000x16", "call": "r", "dtype": "f64", "m": 10000, "n": 16},
        # narrow: a few coefficients over many samples, nearest to memory speed
        {"name": "r f64 16777216x8", "call": "r", "dtype": "f64", "m": 1 << 24, "n": 8},
        # the framework's headline workload
        {"name": "r f64 4194304x32", "call": "r", "dtype": "f64", "m": 1 << 22, "n": 32},
        # the size of the paper's own experiment, ill-conditioned, with a padded leading dimension
        {"name": "r f64 1000000x50 kappa 1e8", "call": "r", "dtype": "f64", "m": 1000000, "n": 50,
         "kappa": 1e8, "pad": 3},
        # the widest that one reduction takes
        {"name": "r f64 4194304x128", "call": "r", "dtype": "f64", "m": 1 << 22, "n": 128},
        # mixed precision: FP32 data (single-precision pipelines), moderately conditioned
        {"name": "r f32 16777216x64 kappa 1e4", "call": "r", "dtype": "f32", "m": 1 << 24, "n": 64,
         "kappa": 1e4},
        # mixed precision: BF16 activations, odd sizes (no aligned leading dimension)
        {"name": "r bf16 1000003x40", "call": "r", "dtype": "bf16", "m": 1000003, "n": 40},
        # many independent problems of all sizes in one call, FP64 and FP32
        {"name": "batch f64 512", "call": "batch", "dtype": "f64", "count": 512, "m_lo": 512,
         "m_hi": 65536, "sizes": 1},
        {"name": "batch f32 1024", "call": "batch", "dtype": "f32", "count": 1024, "m_lo": 512,
         "m_hi": 131072, "sizes": 2},
        # an orthonormal basis of a tall block (block Krylov, randomized range finding)
        {"name": "qr 4194304x32", "call": "qr", "m": 1 << 22, "n": 32},
        # a linear regression, one right-hand side
        {"name": "lstsq 1000000x32 k1", "call": "lstsq", "m": 1000000, "n": 32, "k": 1},
        # a general matrix, by panels
        {"name": "caqr 65536x512", "call": "caqr", "m": 65536, "n": 512},
    ]


def _spread(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi], odd ones among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["r", "r", "r", "mixed", "mixed", "batch", "qr", "lstsq", "caqr"])
    if call == "r":
        n = rng.randint(1, 128)
        c = {"call": "r", "dtype": "f64", "n": n,
             "m": _spread(rng, 10000, min(1 << 24, (1 << 36) // (n * n)))}
        if n > 1 and rng.random() < 0.3:
            c["kappa"] = rng.choice([1e2, 1e4, 1e6, 1e8])
        if rng.random() < 0.3:
            c["pad"] = rng.randint(1, 9)
        return c
    if call == "mixed":
        n = rng.randint(4, 112)
        c = {"call": "r", "dtype": rng.choice(["f32", "bf16"]), "n": n,
             "m": _spread(rng, 20000, (1 << 30) // n)}
        if rng.random() < 0.5:
            c["kappa"] = rng.choice([1e2, 1e4, 1e6])
        return c
    if call == "batch":
        return {"call": "batch", "dtype": rng.choice(["f64", "f32"]),
                "count": _spread(rng, 64, 1024), "m_lo": 512,
                "m_hi": _spread(rng, 4096, 131072), "sizes": rng.randint(10, 1 << 20)}
    if call == "qr":
        n = rng.randint(2, 64)
        return {"call": "qr", "n": n, "m": _spread(rng, 10000, min(1 << 22, (1 << 32) // (n * n)))}
    if call == "lstsq":
        n = rng.randint(2, 64)
        return {"call": "lstsq", "n": n, "k": rng.choice([1, 1, 2, 8, 32]),
                "m": _spread(rng, 10000, min(1 << 22, (1 << 31) // (n * n)))}
    n = _spread(rng, 130, 640)
    return {"call": "caqr", "n": n, "m": _spread(rng, 4 * n, (1 << 34) // (n * n))}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _matrix(case, seed):
    """(storage, A): A the logical (m, n) column-major view of an (n, lda) tensor."""
    m, n, g = case["m"], case["n"], _gen(seed)
    dtype = _DTYPES[case.get("dtype", "f64")]
    store = torch.empty(n, m + case.get("pad", 0), dtype=dtype, device="cuda")
    kappa = case.get("kappa")
    if kappa:
        v, _ = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=torch.float64, device="cuda"))
        k = torch.arange(n, dtype=torch.float64, device="cuda")
        mix = v * torch.pow(torch.tensor(kappa, dtype=torch.float64, device="cuda"), -k / (n - 1))
    for lo in range(0, m, 1 << 22):
        rows = min(1 << 22, m - lo)
        part = torch.randn(n, rows, generator=g, dtype=torch.float64 if kappa or dtype == torch.float64
                           else torch.float32, device="cuda")
        store[:, lo:lo + rows] = mix @ part if kappa else part
    return store, store[:, :m].T


def _batch_sizes(case):
    """Rows log-uniform in [m_lo, m_hi], widths of {8, 16, 32, 64}: the same for every seed."""
    g = torch.Generator().manual_seed(case["sizes"])
    u = torch.rand(case["count"], generator=g, dtype=torch.float64)
    ms = torch.exp(math.log(case["m_lo"]) + u * math.log(case["m_hi"] / case["m_lo"]))
    ns = torch.tensor([8, 16, 32, 64])[torch.randint(0, 4, (case["count"],), generator=g)]
    return [int(round(x)) for x in ms.tolist()], ns.tolist()


def _batch_data(case, seed):
    ms, ns = _batch_sizes(case)
    offs = [0]
    for m, n in zip(ms, ns):
        offs.append(offs[-1] + m * n)
    return torch.randn(offs[-1], generator=_gen(seed), dtype=_DTYPES[case["dtype"]],
                       device="cuda"), ms, ns, offs


def _rhs(case, A, seed):
    """Right-hand sides of a regression: A x0 and noise of a tenth of its size."""
    m, n, k, g = case["m"], case["n"], case["k"], _gen(seed + 7919)
    x0 = torch.randn(n, k, generator=g, dtype=torch.float64, device="cuda")
    noise = torch.randn(k, m, generator=g, dtype=torch.float64, device="cuda")
    return ((A @ x0).T + 0.1 * math.sqrt(n) * noise).contiguous().T


def prepare(case, seed):
    if case["call"] == "batch":
        buf, ms, ns, offs = _batch_data(case, seed)
        roff = [0]
        for n in ns:
            roff.append(roff[-1] + n * n)
        es = buf.element_size()
        f64 = case["dtype"] == "f64"
        return {"call": "batch", "buf": buf, "ptrs": [buf.data_ptr() + es * o for o in offs[:-1]],
                "ms": ms, "ns": ns, "roff": roff,
                "R": torch.empty(roff[-1], dtype=torch.float64, device="cuda"),
                "dtype": tsqr.F64 if f64 else tsqr.F32,
                "prec": tsqr.PREC_F64 if f64 else tsqr.PREC_MIXED}
    store, A = _matrix(case, seed)
    state = {"call": case["call"], "dtype": case.get("dtype", "f64"), "store": store, "A": A}
    if case["call"] == "lstsq":
        state["B"] = _rhs(case, A, seed)
    return state


def run(state):
    call = state["call"]
    if call == "batch":
        return tsqr.tsqr_r_batched(state["ptrs"], state["ms"], state["ns"], state["roff"],
                                   state["R"], dtype=state["dtype"], prec=state["prec"])
    if call == "qr":
        return tsqr.tsqr_qr(state["A"])
    if call == "lstsq":
        return tsqr.tsqr_lstsq(state["A"], state["B"])
    if call == "caqr":
        return tsqr.tsqr_caqr_r(state["A"])
    return tsqr.tsqr_r(state["A"]) if state["dtype"] == "f64" else tsqr.tsqr_r_ex(state["A"])


def _r_flops(m, n):
    return 2.0 * m * n * n - 2.0 * n ** 3 / 3.0


def work(case):
    size = {"f64": 8, "f32": 4, "bf16": 2}[case.get("dtype", "f64")]
    if case["call"] == "batch":
        ms, ns = _batch_sizes(case)
        return {"bytes": sum(size * m * n + 8 * n * n for m, n in zip(ms, ns)),
                "flops": sum(_r_flops(m, n) for m, n in zip(ms, ns))}
    m, n = case["m"], case["n"]
    nbytes, flops = size * m * n + 8 * n * n, _r_flops(m, n)
    if case["call"] == "qr":
        nbytes, flops = nbytes + 8 * m * n, 2 * flops
    if case["call"] == "lstsq":
        k = case["k"]
        nbytes, flops = nbytes + 8 * (m + n) * k, flops + 4.0 * m * n * k
    return {"bytes": nbytes, "flops": flops}


def _signs(r):
    s = torch.sign(torch.diagonal(r))
    return torch.where(s == 0, torch.ones_like(s), s)


def _exact_r(A):
    """R of A in 64 bits: blocks of rows, then the stack of their triangles."""
    m, n = A.shape
    step = max(1 << 18, 2 * n)
    if m > 2 * step:
        parts = [torch.linalg.qr(A[lo:lo + step].double().contiguous(), mode="r")[1]
                 for lo in range(0, m, step)]
        r = torch.linalg.qr(torch.cat(parts), mode="r")[1]
    else:
        r = torch.linalg.qr(A.double().contiguous(), mode="r")[1]
    return (_signs(r)[:, None] * r).triu()


def exact(case, seed):
    if case["call"] == "batch":
        buf, ms, ns, offs = _batch_data(case, seed)
        return torch.cat([_exact_r(buf[o:o + m * n].reshape(n, m).T).T.reshape(-1)
                          for m, n, o in zip(ms, ns, offs)])
    store, A = _matrix(case, seed)
    if case["call"] == "qr":
        q, r = torch.linalg.qr(A.contiguous())
        s = _signs(r)
        return q * s, (s[:, None] * r).triu()
    if case["call"] == "lstsq":
        n, k = case["n"], case["k"]
        r = _exact_r(torch.cat([A, _rhs(case, A, seed)], dim=1))
        x = torch.linalg.solve_triangular(r[:n, :n], r[:n, n:n + k], upper=True)
        return x, r[:n, :n].contiguous()
    return _exact_r(A)
