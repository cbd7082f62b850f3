"""What a user of this library runs, as cases to be timed and checked.

A case names one public entry point of ``paper_2203_02798_gb300``, the sizes
and options of the call, and the distribution of its inputs.  ``listed()``
holds the fixed cases, ``draw(rng)`` one more of the same ranges; ``prepare``
makes what the caller has in hand, ``run`` is one call, ``work`` the bytes and
operations the call cannot do without, and ``exact`` its result in 64 bits
from plain torch (the random draws included: they are a pure function of the
seed and the index, so that they belong to the definition of the result).

Matrices are those of the workloads this library is built for: dense N(0,1)
(with five rows x100, or with columns scaled 10^U(-3,3)), or CSR with each
entry kept with a fixed probability.  Sketches have r = d^2 (at least 4 d)
buckets and k = 2 d Gaussian rows unless a workload names other sizes.
"""
import math

import torch

import paper_2203_02798_gb300 as lsk

DEVICE = "cuda"


def listed():
    return [
        # leverage scores of a small dense matrix in the default precision: 4 MB of input, so
        # that the chain of short launches is what is waited for; d = 50 leaves rows unaligned
        dict(name="lev_small_fp32", op="leverage", fmt="dense", values="outliers", n=20_000, d=50, r=2_500, k=100,
             prec="fp32"),
        # leverage scores of a sparse matrix with two nonzeros a row (the paper's CSR case)
        dict(name="lev_csr_fp32", op="leverage", fmt="csr", density=0.01, n=1_000_000, d=200, r=40_000, k=400,
             prec="fp32"),
        # the headline: BF16 Gaussian stage, TF32 row norms, two passes over 4.1 GB
        dict(name="lev_tall_tf32", op="leverage", fmt="dense", values="colscaled", n=4_000_000, d=256, r=65_536,
             k=512, prec="tf32"),
        # an ordinary dense problem on its own in the mode batches and solvers use
        dict(name="lev_mid_bf16", op="leverage", fmt="dense", values="normal", n=333_333, d=128, r=16_384, k=256,
             prec="bf16"),
        # the CountSketch alone (k = 0 pipelines), a ragged width
        dict(name="cs_ragged", op="cs_sketch", fmt="dense", values="normal", n=1_234_567, d=100, r=10_000),
        # the Gram matrix as the call without options forms it
        dict(name="gram_dense_fp32", op="gram", fmt="dense", values="colscaled", n=1_000_000, d=256, prec="fp32"),
        # the Gram matrix of a sparse matrix (Alg. 5 / 7)
        dict(name="gram_csr", op="gram", fmt="csr", density=0.01, n=1_000_000, d=200, prec="fp32"),
        # squared row norms of A B for a general B as the call without options forms them
        dict(name="rownorms_fp32", op="rownorms", fmt="dense", values="normal", n=750_001, d=200, c=200, prec="fp32"),
        # one served least-squares request, dense and sparse
        dict(name="lsq_dense", op="lsq", fmt="dense", values="normal", n=316_227, d=128),
        dict(name="lsq_csr", op="lsq", fmt="csr", density=0.02, n=500_000, d=256),
        # many independent problems in one call, half dense, half CSR
        dict(name="batch_24", op="batch", count=24, lo=4.0, hi=6.0, spec=3),
        # the one-stage Gaussian sketch of a sparse matrix (Alg. 4)
        dict(name="csrjlt_fp32", op="csrjlt", fmt="csr", density=0.01, n=500_000, d=200, m=400, prec="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["leverage", "leverage", "leverage", "cs_sketch", "gram", "gram", "rownorms", "lsq", "lsq",
                     "batch", "csrjlt"])
    n = _log_int(rng, 1e4, 1e6)
    d = rng.choice([32, 50, 64, 100, 128, 200, 256, rng.randint(17, 256)])
    case = dict(op=op, fmt=rng.choice(["dense", "dense", "csr"]), n=n, d=d)
    if op == "leverage":
        case.update(r=max(d * d, 4 * d), k=2 * d, prec=rng.choice(["fp32", "tf32", "bf16"]))
    elif op == "cs_sketch":
        case.update(r=_log_int(rng, 256, 65_536))
    elif op == "gram":
        case.update(prec=rng.choice(["fp32", "fp32", "bf16"]))
    elif op == "rownorms":
        case.update(c=rng.choice([d, 64, rng.randint(8, 256)]), prec=rng.choice(["fp32", "fp32", "bf16", "tf32"]))
    elif op == "batch":
        return dict(op="batch", count=rng.randint(4, 24), lo=4.0, hi=rng.uniform(5.0, 6.0), spec=rng.randint(4, 999))
    elif op == "csrjlt":
        case.update(fmt="csr", n=min(n, 500_000), m=rng.randint(16, 400), prec=rng.choice(["fp32", "bf16"]))
    if case["fmt"] == "csr":
        case.update(density=round(rng.uniform(0.005, 0.05), 4))
    else:
        case.update(values=rng.choice(["normal", "colscaled", "outliers"]))
    if op == "csrjlt":
        case.update(density=min(case["density"], 0.01))
    return case


# ------------------------------------------------------------------ inputs --
def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _sketch_seed(seed):
    return 7_919 * int(seed) + 2


def _csr(n, d, density, g):
    vs, js, counts = [], [], []
    step = max(1, (1 << 26) // d)
    for i0 in range(0, n, step):
        m = min(step, n - i0)
        rows, cols = torch.nonzero(torch.rand((m, d), generator=g, device=DEVICE) < density, as_tuple=True)
        counts.append(torch.bincount(rows, minlength=m))
        js.append(cols.to(torch.int32))
        vs.append(torch.randn(rows.numel(), generator=g, device=DEVICE))
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
    ptr[1:] = torch.cumsum(torch.cat(counts), 0)
    return lsk.CSR(torch.cat(vs), torch.cat(js), ptr, n, d)


def _matrix(case, g):
    n, d = case["n"], case["d"]
    if case["fmt"] == "csr":
        return _csr(n, d, case["density"], g)
    A = torch.randn((n, d), generator=g, device=DEVICE)
    if case["values"] == "outliers":
        A[:5] *= 100.0
    elif case["values"] == "colscaled":
        A *= 10.0 ** (6.0 * torch.rand(d, generator=g, device=DEVICE) - 3.0)
    return A


def _batch_specs(case):
    """count problems: n = 10^U(lo, hi), d of four widths, the second half CSR."""
    g = torch.Generator()
    g.manual_seed(case["spec"])
    u = torch.rand((case["count"], 3), generator=g, dtype=torch.float64).tolist()
    specs = []
    for p, (a, b, c) in enumerate(u):
        d = (32, 64, 128, 256)[int(4 * b)]
        s = dict(n=int(10.0 ** (case["lo"] + (case["hi"] - case["lo"]) * a)), d=d, r=d * d, k=2 * d, prec="bf16")
        if p < case["count"] // 2:
            s.update(fmt="dense", values="normal")
        else:
            s.update(fmt="csr", density=0.005 + 0.045 * c)
        specs.append(s)
    return specs


def _rows64(A, i0, i1):
    """Rows i0..i1 of A as a dense float64 matrix."""
    if not isinstance(A, lsk.CSR):
        return A[i0:i1].double()
    ptr = A.I[i0:i1 + 1]
    lo, hi = int(ptr[0]), int(ptr[-1])
    rows = torch.repeat_interleave(torch.arange(i1 - i0, device=DEVICE), ptr[1:] - ptr[:-1])
    out = torch.zeros((i1 - i0, A.d), dtype=torch.float64, device=DEVICE)
    out.index_put_((rows, A.J[lo:hi].long()), A.V[lo:hi].double(), accumulate=True)
    return out


def _blocks(A, step=1 << 18):
    n = A.n if isinstance(A, lsk.CSR) else A.shape[0]
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        specs = _batch_specs(case)
        probs = []
        for p, s in enumerate(specs):
            probs.append((_matrix(s, _generator(1_000 * seed + p)), s["r"], s["k"], _sketch_seed(seed) + p))
        return dict(case=case, problems=probs)
    g = _generator(seed)
    state = dict(case=case, A=_matrix(case, g), seed=_sketch_seed(seed))
    if op == "rownorms":
        state["B"] = torch.randn((case["d"], case["c"]), generator=g, device=DEVICE) / math.sqrt(case["d"])
    elif op == "lsq":
        x = torch.randn(case["d"], generator=g, device=DEVICE, dtype=torch.float64)
        b = torch.cat([_rows64(state["A"], i, j) @ x for i, j in _blocks(state["A"])])
        state["b"] = b + 1e-6 * torch.randn(case["n"], generator=g, device=DEVICE, dtype=torch.float64)
    return state


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "batch":
        return lsk.batch_leverage_scores(state["problems"])
    A = state["A"]
    if op == "leverage":
        return lsk.leverage_scores(A, case["r"], case["k"], state["seed"], case["prec"])
    if op == "cs_sketch":
        return lsk.cs_sketch(A, case["r"], state["seed"])
    if op == "gram":
        return lsk.gram(A, prec=case["prec"])
    if op == "rownorms":
        return lsk.rownorms_prod(A, state["B"], prec=case["prec"])
    if op == "csrjlt":
        return lsk.csrjlt(A, case["m"], state["seed"], case["prec"])
    return lsk.sketch_precondition_lsq(A, state["b"])[0]


# -------------------------------------------------------------------- work --
def work(case):
    op = case["op"]
    if op == "batch":
        parts = [work(dict(s, op="leverage")) for s in _batch_specs(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    n, d = case["n"], case["d"]
    if case["fmt"] == "csr":
        nnz = int(n * d * case["density"])
        inp, per_row = 8 * nnz + 8 * (n + 1), nnz / n
    else:
        nnz, inp, per_row = n * d, 4 * n * d, d
    if op == "leverage":
        r, k = case["r"], case["k"]
        norms = n * d * (d + 1) if case["fmt"] == "dense" else 3 * n * per_row * per_row
        return {"bytes": inp + 4 * n, "flops": int(nnz + 2 * k * r * d + k * d * (d + 1) + norms)}
    if op == "cs_sketch":
        return {"bytes": inp + 4 * case["r"] * d, "flops": nnz}
    if op == "gram":
        return {"bytes": inp + 4 * d * d, "flops": int(n * per_row * (per_row + 1))}
    if op == "rownorms":
        c = case["c"]
        prod = 2 * n * d * c if case["fmt"] == "dense" else 3 * n * per_row * per_row + 2 * d * d * c
        return {"bytes": inp + 4 * d * c + 4 * n, "flops": int(prod + 2 * n * c)}
    if op == "csrjlt":
        return {"bytes": inp + 4 * case["m"] * d, "flops": 2 * case["m"] * nnz}
    # least squares: the sketch, then at least one product with A and one with its transpose
    r, k = max(d * d, 4 * d), 2 * d
    return {"bytes": inp + 8 * n + 8 * d, "flops": int(5 * nnz + 2 * k * r * d + k * d * (d + 1))}


# ------------------------------------------------------------------- exact --
def _philox(c0, c1, c2, c3, key):
    """Philox-4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(m, x):
        p, q = x * (m & 0xFFFF), x * (m >> 16)
        return (q + (p >> 16)) >> 16, ((q << 16) + p) & mask

    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _gaussian(rows, c0, c1, stream, key, scale_rows, prec):
    """Columns c0..c1 of the rows x . Gaussian matrix N(0, 1/scale_rows), float64."""
    quads = (rows + 3) // 4
    j = torch.arange(quads, device=DEVICE).view(-1, 1).expand(-1, c1 - c0)
    c = torch.arange(c0, c1, device=DEVICE).view(1, -1).expand(quads, -1)
    w = _philox(c & 0xFFFFFFFF, c >> 32, torch.full_like(c, stream), j, key)
    out = torch.empty((quads, 4, c1 - c0), dtype=torch.float64, device=DEVICE)
    for p in range(2):
        u1 = ((w[2 * p] >> 8) + 1).double() * 2.0 ** -24
        u2 = (w[2 * p + 1] >> 8).double() * 2.0 ** -24
        rad, ang = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
        out[:, 2 * p], out[:, 2 * p + 1] = rad * torch.cos(ang), rad * torch.sin(ang)
    out = out.view(4 * quads, -1)[:rows] / math.sqrt(scale_rows)
    return out if prec == "fp32" else out.float().bfloat16().double()


def _count_sketch(A, d, r, key):
    SA = torch.zeros((r, d), dtype=torch.float64, device=DEVICE)
    for i0, i1 in _blocks(A):
        i = torch.arange(i0, i1, device=DEVICE)
        zero = torch.zeros_like(i)
        w = _philox(i & 0xFFFFFFFF, i >> 32, zero, zero, key)
        sign = (1 - 2 * (w[1] >> 31)).double().view(-1, 1)
        SA.index_add_(0, (w[0] * r) >> 32, _rows64(A, i0, i1) * sign)
    return SA


def _leverage(A, case, key):
    d, r, k = case["d"], case["r"], case["k"]
    SA = _count_sketch(A, d, r, key)
    sketch = torch.zeros((k, d), dtype=torch.float64, device=DEVICE)
    for c0 in range(0, r, 8192):
        c1 = min(r, c0 + 8192)
        sketch += _gaussian(k, c0, c1, 1, key, k, case["prec"]) @ SA[c0:c1]
    R = torch.linalg.qr(sketch, mode="r")[1]
    out = [torch.linalg.solve_triangular(R, _rows64(A, i, j), upper=True, left=False).square().sum(1)
           for i, j in _blocks(A)]
    return torch.cat(out)


def exact(case, seed):
    op, state = case["op"], prepare(case, seed)
    if op == "batch":
        return [_leverage(A, s, key) for s, (A, _, _, key) in zip(_batch_specs(case), state["problems"])]
    A, key, d = state["A"], state["seed"], case["d"]
    if op == "leverage":
        return _leverage(A, case, key)
    if op == "cs_sketch":
        return _count_sketch(A, d, case["r"], key)
    if op == "gram":
        C = torch.zeros((d, d), dtype=torch.float64, device=DEVICE)
        for i, j in _blocks(A):
            rows = _rows64(A, i, j)
            C += rows.T @ rows
        return C
    if op == "rownorms":
        B = state["B"].double()
        return torch.cat([(_rows64(A, i, j) @ B).square().sum(1) for i, j in _blocks(A)])
    if op == "csrjlt":
        C = torch.zeros((case["m"], d), dtype=torch.float64, device=DEVICE)
        for i, j in _blocks(A, 1 << 16):
            C += _gaussian(case["m"], i, j, 3, key, case["m"], case["prec"]) @ _rows64(A, i, j)
        return C
    # least squares: Householder QR of (A b), one refinement on the residual
    rows = torch.cat([_rows64(A, i, j) for i, j in _blocks(A)])
    b = state["b"].view(-1, 1)
    R = torch.linalg.qr(rows, mode="r")[1]

    def seminormal(v):
        y = torch.linalg.solve_triangular(R.T, rows.T @ v, upper=False)
        return torch.linalg.solve_triangular(R, y, upper=True)

    x = seminormal(b)
    for _ in range(2):
        x = x + seminormal(b - rows @ x)
    return x.view(-1)
