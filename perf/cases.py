"""Timed workloads of the noisy-MPO engine, through its public entry points.

Kinds of case:

  circuit  one noisy brickwork circuit from the product state: a new handle,
           every layer applied, the entropies, trace and discarded weight read
           after each (the paper's simulation, Sec. 4.1)
  batch    several such circuits advanced together by the batching form
  sample   output strings drawn from a prepared state by sequential
           conditionals, and their probabilities (Sec. 3.4)
  svd      the truncated SVD of one two-site block theta' (App. A): the work of
           one noisy gate, in the arithmetic of one precision form, and the
           kept block that the two factors stand for
  gemm     the FP64-accurate complex product of the precision form

Singular vectors are fixed only up to phases (and rotations among close
values), so an svd case returns the kept block U X, formed with the
framework's own FP64-accurate product, beside the squared singular values.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2003_13163_gb300 import mpo

DEV = "cuda"


def listed():
    return [
        # n = 8, exact bonds (chi_max = 256 truncates nothing): the smallest
        # factorisations, where launches and waits count
        dict(name="circuit_n8_chi256_fp64", kind="circuit", n=8, chi=256, depth=8, p=0.02, precision="fp64"),
        # the precision form on a short truncated chain
        dict(name="circuit_n12_chi64_mixed", kind="circuit", n=12, chi=64, depth=6, p=0.005, precision="mixed"),
        # an ensemble of circuit instances of uneven length, complex64
        dict(name="batch_k6_chi64_fp32", kind="batch", k=6, n_min=8, n_max=14, chi=64, depth=6, p=0.01,
             precision="fp32"),
        # 2000 output strings of a truncated state
        dict(name="sample_n16_chi64", kind="sample", n=16, chi=64, depth=6, p=0.01, strings=2000, precision="fp64"),
        # one gate's factorisation in the plain form: in the bulk at chi_max = 64,
        # and next to a narrower bond (192) at chi_max = 256
        dict(name="svd_fp64_256x256_chi64", kind="svd", r=256, c=256, cap=64, precision="fp64"),
        dict(name="svd_fp64_768x1024_chi256", kind="svd", r=768, c=1024, cap=256, precision="fp64"),
        # the complex64 form at chi_max = 128
        dict(name="svd_fp32_512x512_chi128", kind="svd", r=512, c=512, cap=128, precision="fp32"),
        # the precision form: odd sides near the end of a chain at chi_max = 150,
        # a bulk gate at chi_max = 256, and one at chi_max = 1024 (the largest)
        dict(name="svd_mixed_577x600_chi150", kind="svd", r=577, c=600, cap=150, precision="mixed"),
        dict(name="svd_mixed_1024x1024_chi256", kind="svd", r=1024, c=1024, cap=256, precision="mixed"),
        dict(name="svd_mixed_4096x4096_chi1024", kind="svd", r=4096, c=4096, cap=1024, precision="mixed"),
        # the precision form's product: the size of a projection at
        # chi_max = 1024, and a ragged one with both operands transposed
        dict(name="gemm_4096x2048x4096", kind="gemm", M=4096, N=2048, K=4096, opA=1, opB=0),
        dict(name="gemm_513x300x1100", kind="gemm", M=513, N=300, K=1100, opA=1, opB=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["circuit", "batch", "sample", "svd", "svd", "svd", "svd", "gemm"])
    if kind == "circuit":
        precision = rng.choice(["fp64", "mixed"])
        return dict(kind=kind, n=rng.choice([6, 8, 10]), chi=rng.choice([16, 32, 48, 64]), depth=rng.randint(3, 6),
                    p=rng.choice([0.005, 0.01, 0.02, 0.05]), precision=precision)
    if kind == "batch":
        return dict(kind=kind, k=rng.randint(2, 6), n_min=rng.choice([6, 8]), n_max=rng.choice([10, 12, 14]),
                    chi=rng.choice([16, 32, 64]), depth=rng.randint(3, 6), p=rng.choice([0.005, 0.01, 0.02, 0.05]),
                    precision="fp32")
    if kind == "sample":
        return dict(kind=kind, n=rng.choice([8, 10, 12, 14, 16]), chi=rng.choice([16, 32, 64]),
                    depth=rng.randint(3, 6), p=rng.choice([0.005, 0.01, 0.02, 0.05]),
                    strings=_log_int(rng, 10, 2000), precision=rng.choice(["fp64", "mixed"]))
    if kind == "gemm":
        return dict(kind=kind, M=_log_int(rng, 64, 4096), N=_log_int(rng, 64, 2048), K=_log_int(rng, 64, 4096),
                    opA=rng.randint(0, 1), opB=rng.randint(0, 1))
    precision = rng.choice(["fp64", "fp32", "mixed", "mixed"])
    r = _log_int(rng, 64, {"fp64": 800, "fp32": 1024, "mixed": 2048}[precision])
    c = min(4096, int(round(r * rng.choice([1.0, 1.0, rng.uniform(1.0, 2.0)]))))
    if precision == "fp64":
        c = min(c, 1024)
    return dict(kind="svd", r=r, c=c, cap=max(1, int(round(r / rng.choice([4, 4, rng.uniform(2.5, 8.0)])))),
                precision=precision)


# ---------------------------------------------------------------- inputs ----
def _bonds(n, parity):
    return range(parity, n - 1, 2)


def _haar_layers(n, depth, rng):
    """depth brickwork layers of Haar-random two-qubit gates: the QR of a
    complex Gaussian with the phase of R's diagonal taken out."""
    layers = []
    for t in range(depth):
        gates = []
        for _ in _bonds(n, t % 2):
            q, r = np.linalg.qr((rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4))) / np.sqrt(2.0))
            gates.append(q * (np.diagonal(r) / np.abs(np.diagonal(r)))[None, :])
        layers.append(np.array(gates, dtype=np.complex128).reshape(-1, 4, 4))
    return layers


def _mix(X, dim, phases):
    """Two rounds of (random phases, unitary DFT) along dim: a dense unitary
    applied to X without forming it."""
    shape = [1, 1]
    shape[dim] = X.shape[dim]
    for ph in phases:
        X = torch.fft.fft(X * ph.reshape(shape), dim=dim, norm="ortho")
    return X


def _theta_parts(case, seed):
    """The unitary mixers and the singular values of a saturated two-site
    block: s_j = exp(-6.9 (j / chi)^0.52) with 2 % scatter, so that the last
    kept value is 1e-3 of the largest and the values fall by 0.05 from j = chi
    to 2 chi, as in the blocks of truncated circuits at chi = 1024."""
    r, c = case["r"], case["c"]
    g = torch.Generator(device=DEV).manual_seed(seed)

    def phases(n):
        return [torch.exp(2j * math.pi * torch.rand(n, dtype=torch.float64, device=DEV, generator=g)) for _ in range(2)]

    left, right = phases(r), phases(c)
    j = torch.arange(r, dtype=torch.float64, device=DEV)
    scatter = 1.0 + 0.02 * (torch.rand(r, dtype=torch.float64, device=DEV, generator=g) - 0.5)
    s = torch.exp(-6.9 * (j / case["cap"]) ** 0.52) * scatter
    return left, right, torch.sort(s, descending=True).values


def _theta(case, parts, keep):
    left, right, s = parts
    X = torch.zeros((case["r"], case["c"]), dtype=torch.complex128, device=DEV)
    X.diagonal()[:keep] = s[:keep].to(torch.complex128)
    return _mix(_mix(X, 0, left), 1, right)


def _operands(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    M, N, K = case["M"], case["N"], case["K"]
    A = torch.randn((K, M) if case["opA"] else (M, K), dtype=torch.complex128, device=DEV, generator=g)
    B = torch.randn((N, K) if case["opB"] else (K, N), dtype=torch.complex128, device=DEV, generator=g)
    # columns of graded size, as the factors of a truncated block have
    A *= torch.logspace(0, -4, A.shape[1], dtype=torch.float64, device=DEV)
    return A, B


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.Generator(np.random.PCG64(seed))
    if kind == "circuit":
        return dict(case=case, layers=_haar_layers(case["n"], case["depth"], rng))
    if kind == "batch":
        n_list = [2 * int(round(v)) for v in np.linspace(case["n_min"] / 2, case["n_max"] / 2, case["k"])]
        per = [_haar_layers(n, case["depth"], rng) for n in n_list]
        return dict(case=case, n_list=n_list, layers=[[q[t] for q in per] for t in range(case["depth"])])
    if kind == "sample":
        m = mpo.MPO(case["n"], case["chi"], case["precision"], centre_only=True)
        for t, gates in enumerate(_haar_layers(case["n"], case["depth"], rng)):
            m.apply_layer(t % 2, gates, case["p"])
        return dict(case=case, mpo=m, uniforms=rng.random((case["strings"], case["n"])))
    if kind == "svd":
        A = _theta(case, _theta_parts(case, seed), case["r"])
        return dict(case=case, A=A.to(torch.complex64) if case["precision"] == "fp32" else A)
    A, B = _operands(case, seed)
    return dict(case=case, A=A, B=B)


# ------------------------------------------------------------------- run ----
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "circuit":
        log = []
        with mpo.MPO(case["n"], case["chi"], case["precision"]) as m:
            for t, gates in enumerate(state["layers"]):
                m.apply_layer(t % 2, gates, case["p"])
                S, trace, discarded = m.entropy()
                log.append([*S, trace, discarded])
        return np.array(log)
    if kind == "batch":
        b = mpo.MPOBatch(state["n_list"], case["chi"], case["precision"])
        log = []
        for t, gates in enumerate(state["layers"]):
            S, trace, discarded = b.apply_layer(t + 1, gates, case["p"])
            log.append(np.concatenate([*S, trace, discarded]))
        b.close()
        return np.array(log)
    if kind == "sample":
        bits, P = state["mpo"].sample(state["uniforms"])
        return {"bits": bits, "P": P, "again": state["mpo"].probability(bits)}
    if kind == "svd":
        U, X, lam2 = mpo.svd_truncated(state["A"], case["cap"], case["precision"])
        kept = mpo.gemm_ex(U.contiguous(), X, 0, 0, "fp32" if case["precision"] == "fp32" else "fp64",
                           0 if case["precision"] == "fp32" else 1)
        return {"kept": kept, "lam2": lam2}
    return mpo.gemm_ex(state["A"], state["B"], case["opA"], case["opB"], "fp64", 1)


# ------------------------------------------------------------------ work ----
def _svd_work(r, c, k, size):
    """Hermitian Gram, dense eigen-decomposition and projection of a truncated
    SVD; the matrix read, the two factors written."""
    return size * (r * c + r * k + k * c), 4.0 * r * r * c + 13.3 * r ** 3 + 8.0 * k * r * c


def _circuit_work(n, chi, depth, size):
    cap = [min(chi, 4 ** min(b, n - b)) for b in range(n + 1)]
    grown = [1] * (n + 1)
    total_b = total_f = 0.0
    for t in range(depth):
        for b in _bonds(n, t % 2):
            cl, cm, cr = grown[b], grown[b + 1], grown[b + 2]
            r, c = 4 * min(cl, cr), 4 * max(cl, cr)
            nb, nf = _svd_work(r, c, min(cap[b + 1], r), size)
            total_b += nb
            total_f += nf + 8.0 * 16 * cl * cr * cm + 2048.0 * cl * cr
            grown[b + 1] = min(cap[b + 1], r)
        for b in range(1, n):           # the Schmidt values of every bond
            nb, nf = _svd_work(grown[b], 4 * grown[b + 1], grown[b], size)
            total_b += nb
            total_f += nf
    return total_b, total_f


def work(case):
    kind = case["kind"]
    size = 8.0 if case.get("precision") == "fp32" else 16.0
    if kind == "circuit":
        b, f = _circuit_work(case["n"], case["chi"], case["depth"], size)
    elif kind == "batch":
        n = 2 * round((case["n_min"] + case["n_max"]) / 4)
        b, f = (case["k"] * x for x in _circuit_work(n, case["chi"], case["depth"], size))
    elif kind == "sample":
        n, chi, S = case["n"], case["chi"], case["strings"]
        cap = [min(chi, 4 ** min(k, n - k)) for k in range(n + 1)]
        sites = sum(4.0 * cap[k] * cap[k + 1] for k in range(n))
        # two continuations per site for the samples, one for the probabilities
        b, f = size * 2 * sites + S * n * 9.0 + 16.0 * S, 3 * 8.0 * S * sites / 4
    elif kind == "svd":
        r, c, k = case["r"], case["c"], case["cap"]
        b, f = _svd_work(r, c, k, size)
        b, f = b + size * r * c, f + 8.0 * r * k * c
    else:
        M, N, K = case["M"], case["N"], case["K"]
        b, f = 16.0 * (M * K + K * N + M * N), 8.0 * M * N * K
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------- exact ----
def _dense_log(case, layers):
    """The same circuit on the dense vectorised density matrix (4^n entries,
    digit 2 i + i' per qubit), in 64 bits: each gate and its depolarising
    noise, then the truncation of the cut between its qubits."""
    n, p = case["n"], case["p"]
    lam = 16.0 * p / 15.0
    t1 = np.zeros(4)
    t1[[0, 3]] = 1.0
    tt = np.outer(t1, t1).reshape(16)
    v = np.zeros(4 ** n, dtype=np.complex128)
    v[0] = 1.0
    log = []
    for t, gates in enumerate(layers):
        discarded = 0.0
        for b, U in zip(_bonds(n, t % 2), gates):
            W = U.reshape(2, 2, 2, 2)
            full = np.einsum("abcd,efgh->aebfcgdh", W, W.conj()).reshape(16, 16)
            full = (1.0 - lam) * full + 0.25 * lam * np.outer(tt, tt)
            x = v.reshape(4 ** b, 16, -1)
            x = np.einsum("xy,ayc->axc", full, x, optimize=True)
            rows = 4 ** (b + 1)
            if min(rows, 4 ** n // rows) > case["chi"]:
                left, s, right = np.linalg.svd(x.reshape(rows, -1), full_matrices=False)
                k = case["chi"]
                discarded += float((s[k:] ** 2).sum() / (s ** 2).sum())
                x = (left[:, :k] * s[:k]) @ right[:k]
            v = np.ascontiguousarray(x).reshape(-1)
        S = []
        for b in range(1, n):
            s = np.linalg.svd(v.reshape(4 ** b, -1), compute_uv=False)
            q = s ** 2 / (s ** 2).sum()
            q = q[q > 0]
            S.append(float(-(q * np.log2(q)).sum()))
        tr = v
        for _ in range(n):
            tr = t1 @ tr.reshape(4, -1)
        log.append([*S, float(tr.reshape(()).real), discarded])
    return np.array(log)


def exact(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        if case["n"] > 8:
            return None                 # minutes as a dense simulation
        return _dense_log(case, prepare(case, seed)["layers"])
    if kind == "svd":
        if case["precision"] == "fp32" and case["r"] > case["c"]:
            return None
        parts = _theta_parts(case, seed)
        k = min(case["cap"], case["r"])
        return {"kept": _theta(case, parts, k), "lam2": (parts[2][:k] ** 2).cpu().numpy()}
    if kind == "gemm":
        A, B = _operands(case, seed)
        return (A.conj().T if case["opA"] else A) @ (B.conj().T if case["opB"] else B)
    return None
