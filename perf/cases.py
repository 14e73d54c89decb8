"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the public Python entry points (which marshal to the C
ABI) with inputs that are already where a program has them: device tensors,
pinned host tensors for the host entry point.  The solver overwrites its
matrices, so a pass that starts from a matrix the program keeps begins with a
device copy of it, as such a program would.

Matrices in float32 take the mixed form, whose eigenvalues carry float32
accuracy; a program with float32 matrices keeps its eigenvalues in float32,
so those passes end with that conversion (float64 matrices: float64).

Inputs follow the recipes of the package's seeded generators, drawn on the
device: semicircle matrices (symmetric N(0,1) / sqrt(n)), Q D Q^T with a
clustered geometric spectrum, SCF-like matrices (Q D Q^T, D uniform in
[-10, 10], plus 1e-3 of a semicircle matrix), N(0,1) bands and tridiagonals.
"""
import concurrent.futures
import math

import numpy as np
import torch

from paper_1604_03703_gb300 import api

DT = {"f32": torch.float32, "f64": torch.float64}
_handle = None


def _h():
    """One handle for the process, as a program keeps it."""
    global _handle
    if _handle is None:
        _handle = api.Handle(0)
    return _handle


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the largest single solve: clustered spectrum, mixed form, the benchmark's band width
        dict(name="eig_f32_n16384_b128", kind="eig", dtype="f32", n=16384, b0=128, matrix="clustered"),
        # a semicircle matrix of half that order, library defaults
        dict(name="eig_f32_n8192", kind="eig", dtype="f32", n=8192, b0=0, matrix="semicircle"),
        # an odd order: no row of the matrix but the first starts on a 16-byte boundary
        dict(name="eig_f32_n2731", kind="eig", dtype="f32", n=2731, b0=0, matrix="scf"),
        # a single small matrix, where the call's latency is the cost
        dict(name="eig_f32_n100", kind="eig", dtype="f32", n=100, b0=0, matrix="semicircle"),
        # the plain FP64 form at an ordinary order, ragged against every tile
        dict(name="eig_f64_n3001", kind="eig", dtype="f64", n=3001, b0=0, matrix="semicircle"),
        # the stage entry points one by one: full-to-band at 32, the halving band stages, bisection
        dict(name="stages_f64_n512_b32", kind="stages", dtype="f64", n=512, b0=32),
        # host buffers in, host eigenvalues out
        dict(name="host_f32_n2048", kind="host", dtype="f32", n=2048, b0=0),
        # many small matrices in one persistent launch, through a kept plan
        dict(name="batch_f32_4096", kind="batch", dtype="f32", count=4096, lo=32, hi=512, draw=3),
        # the same in FP64, fewer of them
        dict(name="batch_f64_500", kind="batch", dtype="f64", count=500, lo=32, hi=512, draw=4),
        # an SCF-like sequence of uneven orders above the one-CTA limit, one call
        dict(name="scf_f32_8", kind="scf", dtype="f32", count=8, lo=1024, hi=3072, draw=5),
        # a banded eigenproblem: band stages down to the tridiagonal, then its eigenvalues
        dict(name="band_f32_n8191_b32", kind="band", dtype="f32", n=8191, b0=32),
        # all eigenvalues of a large tridiagonal at full accuracy
        dict(name="bisect_n16384", kind="bisect", dtype="f64", n=16384, rtol=1e-14),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eig", "eig", "eig", "stages", "host", "batch", "batch", "scf", "band", "bisect"])
    dtype = rng.choice(["f32", "f32", "f64"])
    big = 8192 if dtype == "f32" else 3072
    if kind in ("eig", "host"):
        n = _logint(rng, 64, big if kind == "eig" else big // 2)
        widths = [0, 0] + [w for w in ((16, 32, 64, 128) if dtype == "f32" else (16, 32, 64)) if 4 * w <= n]
        c = dict(kind=kind, dtype=dtype, n=n, b0=rng.choice(widths))
        if kind == "eig":
            c["matrix"] = rng.choice(["semicircle", "scf"] if n <= 4096 else ["semicircle"])
        return c
    if kind == "stages":
        return dict(kind=kind, dtype="f64", n=_logint(rng, 65, 700), b0=rng.choice([8, 16, 32]))
    if kind == "batch":
        lo = _logint(rng, 8, 256)
        return dict(kind=kind, dtype=dtype, count=_logint(rng, 8, 2048 if dtype == "f32" else 400), lo=lo,
                    hi=min(512, 2 * lo + rng.randrange(256)), draw=rng.randrange(1 << 20))
    if kind == "scf":
        lo = rng.randrange(1024, 1537)
        return dict(kind=kind, dtype="f32", count=rng.randrange(2, 8), lo=lo, hi=lo + rng.randrange(64, 1536),
                    draw=rng.randrange(1 << 20))
    if kind == "band":
        return dict(kind=kind, dtype=dtype, n=_logint(rng, 200, 8192 if dtype == "f32" else 2048),
                    b0=rng.choice([8, 16, 32, 64] if dtype == "f32" else [8, 16, 32]))
    return dict(kind="bisect", dtype="f64", n=_logint(rng, 100, 16384), rtol=rng.choice([1e-14, 1e-9]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFF)
    return g


def _semicircle(n, dtype, g):
    L = torch.tril(torch.randn(n, n, generator=g, device="cuda", dtype=dtype))
    return (L + torch.tril(L, -1).T) / math.sqrt(n)


def _qdq(D, dtype, g):
    n = D.numel()
    Q, _ = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=dtype))
    A = (Q * D.to(dtype)[None, :]) @ Q.T
    return (A + A.T) * 0.5


def _matrix(kind, n, dtype, g):
    if kind == "semicircle":
        return _semicircle(n, dtype, g)
    if kind == "scf":
        D = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 20.0 - 10.0
        return _qdq(D, dtype, g) + 1e-3 * _semicircle(n, dtype, g)
    # clustered: magnitudes 10^(-6 + 6 k/(m-1)), random signs, 16 copies each, 1e-10 apart
    m = n // 16
    mag = 10.0 ** (-6.0 + 6.0 * torch.arange(m, device="cuda", dtype=torch.float64) / max(m - 1, 1))
    sgn = torch.where(torch.rand(m, generator=g, device="cuda") < 0.5, -1.0, 1.0).double()
    D = ((sgn * mag)[:, None] + 1e-10 * torch.arange(16, device="cuda", dtype=torch.float64)[None, :]).reshape(-1)
    return _qdq(torch.cat([D, torch.zeros(n - D.numel(), device="cuda", dtype=torch.float64)]), dtype, g)


def _sizes(case):
    """The orders of a batch: part of the case (a batch of other matrices of the same orders is another input)."""
    return [int(m) for m in np.random.default_rng(case["draw"]).integers(case["lo"], case["hi"] + 1, size=case["count"])]


def _views(flat, sizes, off):
    return [flat[o:o + m * m].view(m, m) for m, o in zip(sizes, off)]


def _batch_inputs(case, seed):
    """All matrices in one buffer, each starting on a 256-byte boundary as separate allocations would."""
    dtype, sizes = DT[case["dtype"]], _sizes(case)
    off, total = [], 0
    for m in sizes:
        off.append(total)
        total += (m * m + 63) // 64 * 64
    flat = torch.randn(total, generator=_gen(seed), device="cuda", dtype=dtype)
    scale = torch.tensor([1.0 / math.sqrt(m) for m in sizes], device="cuda", dtype=dtype)
    flat *= torch.repeat_interleave(scale, torch.tensor([(m * m + 63) // 64 * 64 for m in sizes], device="cuda"))
    for A in _views(flat, sizes, off):
        A.copy_(torch.triu(A) + torch.triu(A, 1).T)
    return flat, sizes, off


def _band(case, seed):
    """Packed lower band (n, 2 b): N(0,1) within the band, zeros outside and past the end."""
    n, b = case["n"], case["b0"]
    AB = torch.randn(n, 2 * b, generator=_gen(seed), device="cuda", dtype=DT[case["dtype"]])
    d = torch.arange(2 * b, device="cuda")[None, :]
    j = torch.arange(n, device="cuda")[:, None]
    return AB * ((d <= b) & (j + d < n))


def _tridiagonal(case, seed):
    g = _gen(seed)
    return (torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64),
            torch.randn(case["n"] - 1, generator=g, device="cuda", dtype=torch.float64))


def _halving(b):
    out = [b]
    while out[-1] > 1:
        out.append(out[-1] // 2)
    return out


def _dense(case, seed):
    return _matrix(case.get("matrix", "semicircle"), case["n"], DT[case["dtype"]], _gen(seed))


def prepare(case, seed):
    h, k = _h(), case["kind"]
    s = dict(case=case, h=h, dtype=DT[case["dtype"]])
    if k in ("eig", "stages"):
        s["A"] = _dense(case, seed)
        s["work"] = torch.empty_like(s["A"])
    elif k == "host":
        s["A"] = _dense(case, seed).cpu().pin_memory()
    elif k == "batch":
        s["flat"], sizes, off = _batch_inputs(case, seed)
        s["work"] = torch.empty_like(s["flat"])
        s["lam"] = torch.empty(sum(sizes), dtype=torch.float64, device="cuda")
        outs = list(torch.split(s["lam"], sizes))
        s["plan"] = h.batch_plan(_views(s["work"], sizes, off), outs)
    elif k == "scf":
        g = _gen(seed)
        s["A"] = [_matrix("scf", m, s["dtype"], g) for m in _sizes(case)]
        s["work"] = [torch.empty_like(A) for A in s["A"]]
    elif k == "band":
        s["A"] = _band(case, seed)
        s["work"] = torch.empty_like(s["A"])
        s["widths"] = api.band_schedule(case["n"], case["b0"], 1 if case["dtype"] == "f32" else 0)
    else:
        s["d"], s["e"] = _tridiagonal(case, seed)
    return s


# -------------------------------------------------------------------- a pass
def run(s):
    case, h = s["case"], s["h"]
    k = case["kind"]
    if k == "eig":
        s["work"].copy_(s["A"])
        return h.eigvalsh(s["work"], case["b0"]).to(s["dtype"])
    if k == "host":
        return h.eigvalsh_host(s["A"], case["b0"]).to(s["dtype"])
    if k == "batch":
        s["work"].copy_(s["flat"])
        s["plan"].run()
        return s["lam"].to(s["dtype"])
    if k == "scf":
        for w, A in zip(s["work"], s["A"]):
            w.copy_(A)
        return torch.cat(h.eigvalsh_batched(s["work"])).to(s["dtype"])
    if k == "bisect":
        return h.tridiag_bisect(s["d"], s["e"], case["rtol"])
    s["work"].copy_(s["A"])
    if k == "stages":
        band = h.full_to_band(s["work"], case["b0"])
        AB = band.clone()
        widths = _halving(case["b0"])
    else:
        AB, widths = s["work"], s["widths"]
    for b, hh in zip(widths[:-1], widths[1:]):
        h.band_to_band(AB, b, hh)
    d, e = h.band_tridiag(AB)
    lam = h.tridiag_bisect(d, e, 1e-14 if case["dtype"] == "f64" else 1e-9)
    # (the tridiagonal of a float32 band depends on its rounding, its eigenvalues do not)
    return [band, d, e, lam] if k == "stages" else lam.to(s["dtype"])


# -------------------------------------------------------------------- work
def _bisect_flops(n, rtol):
    """Sturm steps of 3 operations: log2(1/rtol) counts an eigenvalue, the first log2(n) of them shared."""
    return 3.0 * n * n * max(1.0, math.log2(1.0 / rtol) - math.log2(max(n, 2)))


def work(case):
    es, k = (4 if case["dtype"] == "f32" else 8), case["kind"]
    rtol = case.get("rtol", 1e-14 if case["dtype"] == "f64" else 1e-9)
    if k in ("batch", "scf"):
        sizes = _sizes(case)
        return {"bytes": sum(es * m * (m + 1) / 2 + es * m for m in sizes), "flops": sum(4.0 * m ** 3 / 3 for m in sizes)}
    n = case["n"]
    if k == "bisect":
        return {"bytes": 8.0 * (2 * n - 1) + 8.0 * n, "flops": _bisect_flops(n, rtol)}
    if k == "band":
        # Givens-like reduction of a band: about 6 n^2 b, then the eigenvalues
        return {"bytes": es * n * (case["b0"] + 1.0) + es * n, "flops": 6.0 * n * n * case["b0"] + _bisect_flops(n, rtol)}
    extra = es * n * (case["b0"] + 1.0) + 8.0 * 2 * n if k == "stages" else 0.0
    return {"bytes": es * n * (n + 1) / 2.0 + es * n + extra, "flops": 4.0 * n ** 3 / 3}


# ------------------------------------------------------------------- exact
def _np_eigs(mats):
    """Eigenvalues of many small matrices on the host cores, largest first."""
    with concurrent.futures.ThreadPoolExecutor(16) as ex:
        return list(ex.map(np.linalg.eigvalsh, mats))


def exact(case, seed):
    """The eigenvalues of the very matrices that `run` gets, in 64 bits."""
    k = case["kind"]
    if k == "batch":
        flat, sizes, off = _batch_inputs(case, seed)
        host = flat.double().cpu().numpy()
        return torch.from_numpy(np.concatenate(_np_eigs([host[o:o + m * m].reshape(m, m) for m, o in zip(sizes, off)])))
    if k == "scf":
        g = _gen(seed)
        return torch.cat([torch.linalg.eigvalsh(_matrix("scf", m, DT[case["dtype"]], g).double()) for m in _sizes(case)])
    if k == "bisect":
        d, e = _tridiagonal(case, seed)
        return torch.linalg.eigvalsh(torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1))
    if k == "band":
        AB = _band(case, seed).double()
        n = case["n"]
        A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        for dd in range(min(case["b0"] + 1, n)):
            A.diagonal(-dd).copy_(AB[: n - dd, dd])
        return torch.linalg.eigvalsh(A, UPLO="L")
    lam = torch.linalg.eigvalsh(_dense(case, seed).double())
    return [None, None, None, lam] if k == "stages" else lam
