"""The work that users of this library have it do, as cases to be timed.

Every case is one call (or one fit with the calls around it) through the public binding
``paper_2606_23274_gb300.ttfit``, at the sizes of this repository's workloads, tests and
benchmark extras:

* ``svd``      tt_svd_truncated: the factorisation of one two-site tensor on its own (FP64);
* ``product``  tt_mpo_naive_product: the exact per-site product of two MPOs (FP64 or FP32);
* ``zipup``    tt_mpo_zipup: the one-pass contraction of two MPOs (FP64);
* ``grad``     tt_mpo_grad: value and gradients of ||X - AB||^2 or <X, AB> (FP64, FP32, 3xTF32);
* ``fit``      a complete FP64 fit: create, sweeps, export of C and of its bond spectra, destroy;
* ``batch``    FP64 fits of several uneven pairs at once, in the inverse gauge;
* ``mixed``    the default schedule to convergence (one 3xTF32 sweep, then FP64-class sweeps with
               BF16 digit products), and the gradient of <C, AB> at the fitted C, which is how C is
               used further in a training loop. C's cores are unique only up to the basis of
               near-degenerate singular pairs; its spectra and that gradient depend on the
               operator alone.

Fits are exported in FP32, as a caller that goes on in FP32 takes them.
"""
import math

import torch

from paper_2606_23274_gb300 import ttfit
from paper_2606_23274_gb300.synth import kron_sum_mpo

OVERSAMPLE = 10
TOL = 1e-8        # convergence threshold of the mixed schedule
MAX_SWEEPS = 14


def listed():
    return [
        # one bond of a short chain: the smallest call, where launches and allocation count
        {"name": "svd_24x16", "kind": "svd", "m": 24, "n": 16, "chi": 12, "tau": 0.0, "floor": 1e-4},
        # a wide window of ragged bonds, truncated by tolerance
        {"name": "svd_101x203", "kind": "svd", "m": 101, "n": 203, "chi": 101, "tau": 1e-3, "floor": 1e-5},
        # the largest factorisation of an exact chi = 64 fit: a 256 x 256 window
        {"name": "svd_256x256", "kind": "svd", "m": 256, "n": 256, "chi": 64, "tau": 0.0, "floor": 1e-4},
        # exact product of two mid-size MPOs: bound by writing C
        {"name": "product_fp32_L8_48x40", "kind": "product", "L": 8, "chi_a": 48, "chi_b": 40, "dtype": "float32"},
        # one-pass contraction as an estimate or an initial guess
        {"name": "zipup_L20_chi64", "kind": "zipup", "L": 20, "chi": 64, "update": "rsvd"},
        # gradient of a short chain in FP64 (as a check, or inside an optimiser's line search)
        {"name": "grad_inner_fp64_L8_chi12", "kind": "grad", "L": 8, "chi": 12, "chi_x": 12, "target": "inner",
         "precision": "fp64"},
        # gradient against a narrower weight MPO, FP32, on the long chain of the benchmark's adjoint
        {"name": "grad_inner_fp32_L32_chi96", "kind": "grad", "L": 32, "chi": 96, "chi_x": 32, "target": "inner",
         "precision": "fp32"},
        # the least-squares gradient with its four-layer environments, tensor-core products
        {"name": "grad_residual_tf32x3_L16_chi48", "kind": "grad", "L": 16, "chi": 48, "chi_x": 48,
         "target": "residual", "precision": "tf32x3"},
        # an accurate fit of a short chain, exact two-site update
        {"name": "fit_fp64_L12_chi32", "kind": "fit", "L": 12, "K": 32, "chi": 32, "update": "svd", "gauge": "site",
         "sweeps": 2},
        # many small independent fits side by side
        {"name": "batch_fp64_8_pairs", "kind": "batch", "pairs": 8, "L_lo": 8, "L_hi": 16, "chi_lo": 6, "chi_hi": 16,
         "sweeps": 3},
        # the default schedule on a mid-size chain
        {"name": "mixed_L20_chi64", "kind": "mixed", "L": 20, "chi": 64},
        # the default schedule on the benchmark's chain
        {"name": "mixed_L30_chi128", "kind": "mixed", "L": 30, "chi": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["svd", "svd", "product", "zipup", "grad", "grad", "fit", "batch", "mixed", "mixed"])
    if kind == "svd":
        m, n = _log_int(rng, 8, 320), _log_int(rng, 8, 320)
        if min(m, n) > 256:
            m = 256
        return {"kind": kind, "m": m, "n": n, "chi": rng.randint(1, min(m, n)), "tau": rng.choice([0.0, 1e-3]),
                "floor": 10.0 ** rng.uniform(-5, -1)}
    if kind == "product":
        return {"kind": kind, "L": rng.randint(3, 12), "chi_a": _log_int(rng, 4, 40), "chi_b": _log_int(rng, 4, 40),
                "dtype": rng.choice(["float32", "float64"])}
    if kind == "zipup":
        return {"kind": kind, "L": rng.randint(8, 20), "chi": _log_int(rng, 12, 64), "update": "rsvd"}
    if kind == "grad":
        target = rng.choice(["inner", "residual"])
        precision = rng.choice(["fp64", "fp32", "tf32x3"])
        if target == "residual":
            chi = _log_int(rng, 8, 14 if precision == "fp64" else 32)
            return {"kind": kind, "L": rng.randint(6, 16), "chi": chi, "chi_x": chi, "target": target,
                    "precision": precision}
        return {"kind": kind, "L": rng.randint(6, 32), "chi": _log_int(rng, 8, 24 if precision == "fp64" else 96),
                "chi_x": _log_int(rng, 8, 32), "target": target, "precision": precision}
    if kind == "fit":
        K = rng.randint(12, 32)
        return {"kind": kind, "L": rng.randint(8, 12), "K": K, "chi": rng.randint(8, K),
                "update": rng.choice(["svd", "rsvd"]), "gauge": rng.choice(["site", "inverse"]), "sweeps": 2}
    if kind == "batch":
        lo, clo = rng.randint(8, 12), rng.randint(6, 10)
        return {"kind": kind, "pairs": rng.randint(2, 8), "L_lo": lo, "L_hi": rng.randint(lo, 16), "chi_lo": clo,
                "chi_hi": rng.randint(clo, 16), "sweeps": rng.randint(2, 3)}
    # (a chain much shorter than the benchmark's does not settle at wide bonds: its sketches keep deciding C)
    return {"kind": "mixed", "L": rng.randint(22, 30), "chi": rng.randint(56, 128)}


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + int(stream)) % (1 << 62))
    return g


def _random_mpo(L, d, chi, seed, stream, dtype):
    """Gaussian cores whose product keeps a norm of about 1, whatever the length."""
    g = _gen(seed, stream)
    bonds = [1] + [chi] * (L - 1) + [1]
    return [(torch.randn(bonds[l], d, d, bonds[l + 1], generator=g, device="cuda", dtype=torch.float64)
             / (d * math.sqrt(chi))).to(dtype) for l in range(L)]


def _kron_pair(L, K, seed):
    return tuple([torch.from_numpy(x).to("cuda") for x in kron_sum_mpo(L, K, seed, w)] for w in (0, 1))


def _batch_sizes(case):
    """Lengths and bonds of a batch's pairs, spread over their ranges."""
    n = case["pairs"]
    at = [i / max(1, n - 1) for i in range(n)]
    Ls = [case["L_lo"] + round(t * (case["L_hi"] - case["L_lo"])) for t in at]
    chis = [case["chi_hi"] - round(t * (case["chi_hi"] - case["chi_lo"])) for t in at]
    return Ls, chis


def _matrix(case, seed):
    """A matrix with singular values decaying about geometrically from 1 to `floor`, as a window's do."""
    m, n = case["m"], case["n"]
    r = min(m, n)
    g = _gen(seed, 0)
    U, _ = torch.linalg.qr(torch.randn(m, r, generator=g, device="cuda", dtype=torch.float64))
    V, _ = torch.linalg.qr(torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64))
    at = torch.arange(r, device="cuda", dtype=torch.float64) / max(1, r - 1)
    jitter = 0.25 * torch.rand(r, generator=g, device="cuda", dtype=torch.float64) / max(1, r - 1)
    return (U * (case["floor"] ** (at + jitter))) @ V.T


GRAD_DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "tf32x3": torch.float32}


def prepare(case, seed):
    k = case["kind"]
    if k == "svd":
        return {"case": case, "M": _matrix(case, seed)}
    if k == "product":
        dt = getattr(torch, case["dtype"])
        return {"case": case, "A": _random_mpo(case["L"], 2, case["chi_a"], seed, 0, dt),
                "B": _random_mpo(case["L"], 2, case["chi_b"], seed, 1, dt)}
    if k == "grad":
        dt = GRAD_DTYPE[case["precision"]]
        return {"case": case, "A": _random_mpo(case["L"], 2, case["chi"], seed, 0, dt),
                "B": _random_mpo(case["L"], 2, case["chi"], seed, 1, dt),
                "X": _random_mpo(case["L"], 2, case["chi_x"], seed, 2, dt)}
    if k == "batch":
        Ls, chis = _batch_sizes(case)
        pairs = [_kron_pair(L, c, seed * 64 + i) for i, (L, c) in enumerate(zip(Ls, chis))]
        return {"case": case, "pairs": pairs, "chis": chis}
    A, B = _kron_pair(case["L"], case["K"] if k == "fit" else case["chi"], seed)
    return {"case": case, "A": A, "B": B, "seed": seed % 1000}


def _flat(tensors):
    return torch.cat([t.reshape(-1) for t in tensors])


def _export(f):
    """C (FP32 cores, one vector) and the spectra of its bonds."""
    C = f.result(torch.float32)
    lam = torch.cat([torch.from_numpy(s) for s in f.lambdas()]).float()
    return C, lam


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "svd":
        U, S, Vt, kept = ttfit.tt_svd_truncated(state["M"], c["chi"], c["tau"])
        return {"U": U, "S": S, "Vt": Vt, "k": kept}
    if k == "product":
        return ttfit.tt_mpo_naive_product(state["A"], state["B"])
    if k == "zipup":
        C = ttfit.tt_mpo_zipup(state["A"], state["B"], c["chi"], 0.0, update=c["update"], oversample=OVERSAMPLE,
                               seed=state["seed"], precision="fp64", dtype=torch.float32)
        return {"C": _flat(C)}
    if k == "grad":
        v, gA, gB = ttfit.tt_mpo_grad(state["A"], state["B"], state["X"], c["target"], c["precision"])
        return {"value": v, "gA": _flat(gA), "gB": _flat(gB)}
    if k == "fit":
        f = ttfit.tt_fit_create(state["A"], state["B"], c["chi"], 0.0, c["gauge"], update=c["update"],
                                oversample=OVERSAMPLE, seed=state["seed"], precision="fp64", conv_tol=0.0)
        rep = f.sweep(c["sweeps"])
        C, lam = _export(f)
        f.destroy()
        return {"C": _flat(C), "lambda": lam, "norm2": rep["norm2_C"]}
    if k == "batch":
        fits = ttfit.tt_fit_create_batched(state["pairs"], state["chis"], 0.0, "inverse", update="rsvd", oversample=4,
                                           seed=7, precision="fp64", conv_tol=0.0)
        reps = ttfit.tt_fit_sweep_batched(fits, c["sweeps"])
        out = []
        for f, rep in zip(fits, reps):
            C, lam = _export(f)
            f.destroy()
            out.append({"C": _flat(C), "lambda": lam, "norm2": rep["norm2_C"]})
        return out
    f = ttfit.tt_fit_create(state["A"], state["B"], c["chi"], TOL, "site", update="rsvd", oversample=OVERSAMPLE,
                            seed=state["seed"], precision="tf32x3")
    rep = f.sweep(1)
    f.set_precision("bf16_split", fast_factor=1)
    while rep["sweeps_done"] < MAX_SWEEPS:
        rep = f.sweep(1)
        if rep["converged"]:
            break
    C, lam = _export(f)
    f.destroy()
    A, B = ([x.float() for x in M] for M in (state["A"], state["B"]))
    v, gA, gB = ttfit.tt_mpo_grad(A, B, C, "inner", "tf32x3")
    return {"lambda": lam, "norm2": rep["norm2_C"], "value": v, "gA": _flat(gA), "gB": _flat(gB)}


# --------------------------------------------------------------------------- work
def _bonds(L, chi, dd=4):
    """Bonds of an MPO trimmed to its rank bound (d d' = dd per site)."""
    return [min(chi, dd ** min(l, L - l, 12)) for l in range(L + 1)]


def _sizes(bonds, dd=4):
    return sum(bonds[l] * dd * bonds[l + 1] for l in range(len(bonds) - 1))


def _window_flops(L, a, b, c, update, ks):
    """One sweep: a fresh half, the two-site tensor, its factorisation and one environment per window (d = 2)."""
    fl = 0.0
    for l in range(L - 1):
        m, n = 4 * c[l], 4 * c[l + 2]
        fl += 2.0 * c[l] * b[l] * a[l] * 4 * a[l + 1] + 2.0 * c[l] * 2 * a[l + 1] * b[l] * 2 * 2 * b[l + 1]
        fl += 2.0 * m * n * a[l + 1] * b[l + 1]
        fl += 2.0 * c[l + 1] * m * a[l + 1] * b[l + 1]
        r = min(m, n)
        k = ks if update == "rsvd" and ks < r else r
        fl += 4.0 * m * n * k + 4.0 * (m + n) * k * k if k < r else 8.0 * max(m, n) * r * r
    return fl


def _grad_flops(L, a, b, x, four):
    """Three-layer environments from both sides and the two holes (d = 2); the four-layer ones too if `four`."""
    fl = 0.0
    for l in range(L):
        step = 8.0 * b[l] * x[l] * a[l] * a[l + 1] + 16.0 * x[l] * a[l + 1] * b[l] * b[l + 1]
        step += 8.0 * a[l + 1] * b[l + 1] * x[l] * x[l + 1]
        fl += 4 * step
        if four:
            # the four contractions of one step: A, B, then A, B of the other copy
            step = 8.0 * b[l] * a[l] * b[l] * a[l] * a[l + 1] + 16.0 * a[l] * b[l] * a[l + 1] * b[l] * b[l + 1]
            step += 16.0 * b[l] * a[l + 1] * b[l + 1] * a[l] * a[l + 1]
            step += 8.0 * a[l + 1] * b[l + 1] * a[l + 1] * b[l] * b[l + 1]
            fl += 4 * step
    return fl


def work(case):
    k = case["kind"]
    if k == "svd":
        m, n = case["m"], case["n"]
        r = min(m, n)
        return {"bytes": 8 * (m * n + m * r + r + r * n), "flops": 8.0 * max(m, n) * r * r}
    if k == "product":
        L, e = case["L"], 8 if case["dtype"] == "float64" else 4
        a, b = ([1] + [case[c]] * (L - 1) + [1] for c in ("chi_a", "chi_b"))
        out = sum(4 * a[l] * b[l] * a[l + 1] * b[l + 1] for l in range(L))
        return {"bytes": e * (_sizes(a) + _sizes(b) + out), "flops": 4.0 * out}
    if k == "zipup":
        L = case["L"]
        a = c = _bonds(L, case["chi"])
        ks = case["chi"] + OVERSAMPLE
        fl = 0.0
        for l in range(L):
            m, n = a[l] * a[l], 4 * c[l + 1]
            fl += 2.0 * 4 * a[l] * a[l + 1] * a[l + 1] * c[l + 1] + 2.0 * m * n * 2 * a[l + 1]
            fl += 2.0 * m * n * (2 * min(ks, n) + c[l])
        return {"bytes": 8 * 2 * _sizes([1] + [case["chi"]] * (L - 1) + [1]) + 4 * _sizes(c), "flops": fl}
    if k == "grad":
        L, e = case["L"], 8 if case["precision"] == "fp64" else 4
        a, x = ([1] + [case[c]] * (L - 1) + [1] for c in ("chi", "chi_x"))
        return {"bytes": e * (4 * _sizes(a) + _sizes(x)),
                "flops": _grad_flops(L, a, a, x, case["target"] == "residual")}
    if k == "batch":
        by = fl = 0.0
        for L, chi in zip(*_batch_sizes(case)):
            a = _bonds(L, chi)
            fl += case["sweeps"] * _window_flops(L, a, a, a, "rsvd", chi + 4)
            by += 8 * 2 * _sizes([1] + [chi] * (L - 1) + [1]) + 4 * (_sizes(a) + sum(a))
        return {"bytes": by, "flops": fl}
    L, chi = case["L"], case["chi"]
    K = case["K"] if k == "fit" else chi
    full, a, c = [1] + [K] * (L - 1) + [1], _bonds(L, K), _bonds(L, chi)
    by = 8 * 2 * _sizes(full) + 4 * (_sizes(c) + sum(c))
    if k == "fit":
        return {"bytes": by, "flops": case["sweeps"] * _window_flops(L, a, a, c, case["update"], chi + OVERSAMPLE)}
    fl = 3 * _window_flops(L, a, a, c, "rsvd", chi + OVERSAMPLE) + _grad_flops(L, full, full, c, False)
    return {"bytes": by + 4 * 2 * _sizes(full), "flops": fl}


# --------------------------------------------------------------------------- exact values
def _exact_svd(case, seed):
    U, S, Vt = torch.linalg.svd(_matrix(case, seed).cpu(), full_matrices=False)
    at = U.abs().argmax(dim=0)
    sign = torch.where(U[at, torch.arange(U.shape[1])] < 0, -1.0, 1.0).double()
    tail = torch.sqrt(torch.flip(torch.cumsum(torch.flip(S * S, [0]), 0), [0]))  # tail[j]: what keeping j leaves out
    k = len(S)
    if case["tau"] > 0:
        small = (tail <= case["tau"] * tail[0]).nonzero()
        k = int(small[0]) if len(small) else k
    k = max(1, min(k, case["chi"], int((S > 1e-13 * S[0]).sum())))
    return {"U": U * sign, "S": S, "Vt": Vt * sign[:, None], "k": k}


def _inner(X, A, B):
    E = torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")
    for a, b, x in zip(A, B, X):
        T = torch.einsum("abc,asux->bcsux", E, a)
        T = torch.einsum("bcsux,buty->csxty", T, b)
        E = torch.einsum("csxty,cstz->xyz", T, x)
    return E.reshape(())


def _norm2(A, B):
    E = torch.ones(1, 1, 1, 1, dtype=torch.float64, device="cuda")
    for a, b in zip(A, B):
        T = torch.einsum("abpq,asux->bpqsux", E, a)
        T = torch.einsum("bpqsux,buty->pqsxty", T, b)
        T = torch.einsum("pqsxty,psvz->qxtyvz", T, a)
        E = torch.einsum("qxtyvz,qvtw->xyzw", T, b)
    return E.reshape(())


def _exact_grad(case, seed):
    s = prepare(case, seed)
    A, B, X = ([t.double() for t in s[k]] for k in ("A", "B", "X"))
    for t in A + B:
        t.requires_grad_(True)
    v = _inner(X, A, B)
    if case["target"] == "residual":
        xx = torch.ones(1, 1, dtype=torch.float64, device="cuda")
        for x in X:
            xx = torch.einsum("cstz,cstw->zw", torch.einsum("cd,dstz->cstz", xx, x), x)
        v = xx.reshape(()) - 2 * v + _norm2(A, B)
    g = torch.autograd.grad(v, A + B)
    return {"value": float(v.detach()), "gA": _flat(g[:len(A)]), "gB": _flat(g[len(A):])}


def exact(case, seed):
    k = case["kind"]
    if k == "svd":
        return _exact_svd(case, seed)
    if k == "product":
        s = prepare(case, seed)
        return [torch.einsum("isuj,kutl->ikstjl", a.double(), b.double())
                .reshape(a.shape[0] * b.shape[0], 2, 2, a.shape[3] * b.shape[3]) for a, b in zip(s["A"], s["B"])]
    if k == "grad":
        return _exact_grad(case, seed)
    return None  # a sketch, a truncation and a number of sweeps decide what these return
