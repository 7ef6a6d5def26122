"""The work a user of this library has it do, as timed cases.

Each case is one call of a public entry point (`zolo_dgemm`, `zolo_pd`,
`zolo_pd_batched`, `zolo_svd`) with the library's default kernel rules, on
seeded synthetic inputs resident on the GPU: A = U diag(sigma) V^T with Haar U
and V and sigma geometric from 1 to 1/kappa, as the repository's workloads draw
them (paper_1806_06204_gb300/synth.py), here drawn on the device.

`guard` is how far the caller's lower bound beta lies below sigma_min: the l_0 =
beta / alpha of a call, which fixes r, the number of iterations and their forms,
is 1 / (kappa guard) and spans 1e-1 .. 1e-12 as the repository's batch does,
while the spectra themselves stay in a range (kappa <= 1e4; 1e3 for the singular
vectors) where Q_p, U and V are determined to far better than the rounding of
any path.
"""
import math
import random

import torch

from paper_1806_06204_gb300 import binding as zb

PREC = {"fp64": zb.ZOLO_FP64, "bf16": zb.ZOLO_SPLIT_BF16, "fp16": zb.ZOLO_SPLIT_FP16,
        "fp8": zb.ZOLO_SPLIT_FP8}
SLICES = {"fp64": 0, "bf16": 9, "fp16": 8, "fp8": 11}   # the FP64-grade slice counts

_HANDLE = None


def _handle():
    """One handle for the process, as a program keeps it."""
    global _HANDLE
    if _HANDLE is None:
        _HANDLE = zb.Handle(torch.cuda.current_device())
    return _HANDLE


def listed():
    return [
        # the building block on a small problem: latency of one call
        dict(name="gemm_fp64_96x64x200", kind="gemm", prec="fp64", m=96, n=64, k=200,
             ta=0, tb=0),
        # the large square product the split path is for
        dict(name="gemm_bf16_4096", kind="gemm", prec="bf16", m=4096, n=4096, k=4096, ta=0, tb=0),
        # ragged sizes, a transposed operand
        dict(name="gemm_fp16_1000x1537x777t", kind="gemm", prec="fp16", m=1000, n=1537, k=777,
             ta=1, tb=0),
        # the Gram shape of a tall matrix: a long inner dimension, a small output
        dict(name="gemm_fp8_512x512x16384t", kind="gemm", prec="fp8", m=512, n=512, k=16384,
             ta=1, tb=0),
        # one small matrix in plain FP64 at l_0 = 1e-8, r = 3: QR and two Cholesky iterations
        dict(name="pd_fp64_256", kind="pd", prec="fp64", m=256, n=256, r=3, kappa=1e4, guard=1e4,
             ns=0, auto=0),
        # a mid-size matrix in plain FP64, r = 6
        dict(name="pd_fp64_1024", kind="pd", prec="fp64", m=1024, n=1024, r=6, kappa=1e4,
             guard=1e4, ns=0, auto=0),
        # a ragged matrix, nothing known about its spectrum: alpha, beta and r from the library
        dict(name="pd_bf16_1300x1000_auto", kind="pd", prec="bf16", m=1300, n=1000, r=0, kappa=1e3,
             guard=1.0, ns=0, auto=1),
        # the large square decomposition: l_0 = 1e-12, r = 8, the final Newton-Schulz step
        dict(name="pd_fp16_4096", kind="pd", prec="fp16", m=4096, n=4096, r=8, kappa=1e3,
             guard=1e9, ns=1, auto=0),
        # a tall panel (least-squares, orthogonalisation)
        dict(name="pd_bf16_8192x512", kind="pd", prec="bf16", m=8192, n=512, r=6, kappa=1e3,
             guard=1e5, ns=1, auto=0),
        # many matrices of uneven sizes and spectra in one call
        dict(name="batch_bf16_48", kind="batch", prec="bf16", count=48, nmin=64, nmax=1024,
             pick=1, ns=1),
        # the whole SVD of a small and of a mid-size matrix
        dict(name="svd_fp64_256", kind="svd", prec="fp64", m=256, n=256, r=3, kappa=1e3, guard=1e5),
        dict(name="svd_fp64_1024", kind="svd", prec="fp64", m=1024, n=1024, r=6, kappa=1e3,
             guard=1e5),
    ]


def draw(rng):
    """One more case: the same kinds over their whole ranges."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["gemm", "gemm", "pd", "pd", "pd", "batch", "svd"])
        prec = rng.choice(["fp64", "bf16", "bf16", "fp16", "fp16", "fp8"])
        if kind == "gemm":
            # any shape the iterations form, from block factors to trailing updates
            c = dict(kind=kind, prec=prec, m=size(32, 8192), n=size(32, 8192), k=size(32, 16384),
                     ta=rng.randrange(2), tb=rng.randrange(2))
        elif kind == "pd":
            n = size(48, 3072)
            m = n if rng.random() < 0.5 else size(n, 16 * n)
            kappa = 10.0 ** rng.uniform(1, 4)
            auto = int(rng.random() < 0.25)
            guard = 1.0 if auto or rng.random() < 0.3 else 10.0 ** rng.uniform(0, 12 - math.log10(kappa))
            c = dict(kind=kind, prec=prec, m=m, n=n, r=rng.choice([0, 0, 2, 3, 6, 8]), kappa=kappa,
                     guard=guard, ns=rng.randrange(2), auto=auto)
        elif kind == "batch":
            nmax = size(96, 1024)
            c = dict(kind=kind, prec=prec, count=size(8, 64), nmin=rng.randrange(48, nmax), nmax=nmax,
                     pick=rng.randrange(1 << 20), ns=rng.randrange(2))
        else:
            n = size(32, 1024)
            c = dict(kind=kind, prec="fp64", m=n if rng.random() < 0.5 else size(n, 4 * n), n=n,
                     r=rng.choice([0, 3, 6]), kappa=10.0 ** rng.uniform(1, 3),
                     guard=10.0 ** rng.uniform(0, 6))
        # no more than the largest listed case (about 4.5e12 modelled flops on the split path),
        # the FP64 pipe being several times slower
        if work(c)["flops"] <= (2.5e11 if c["prec"] == "fp64" else 2.5e12):
            return c


# ------------------------------------------------------------------ the inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(rows, cols, g):
    """rows x cols, column-major."""
    return torch.randn(cols, rows, dtype=torch.float64, device="cuda", generator=g).t()


def _haar(m, n, g):
    q, r = torch.linalg.qr(torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g))
    d = torch.sign(torch.diagonal(r))
    d[d == 0] = 1.0
    return q * d


def _matrix(m, n, kappa, g):
    s = torch.logspace(0, -math.log10(kappa), n, dtype=torch.float64, device="cuda")
    U, V = _haar(m, n, g), _haar(n, n, g)
    return (V @ (U * s).t()).t()   # A = U diag(s) V^T, column-major


def _factors(c, g):
    """The operands of a product as stored (before any transpose)."""
    m, n, k = c["m"], c["n"], c["k"]
    A = _randn(k, m, g) if c["ta"] else _randn(m, k, g)
    return A, _randn(n, k, g) if c["tb"] else _randn(k, n, g)


def _members(c):
    """The sizes, spectra and l_0 of a batch's matrices, fixed by the case."""
    rng = random.Random(c["pick"])
    out = []
    for _ in range(c["count"]):
        n = rng.randint(c["nmin"], c["nmax"])
        kappa = 10.0 ** rng.uniform(1, 4)
        out.append((n, kappa, 10.0 ** rng.uniform(0, 12 - math.log10(kappa))))
    return out


def prepare(case, seed):
    g = _generator(seed)
    kind, prec = case["kind"], PREC[case["prec"]]
    st = {"kind": kind, "h": _handle(), "prec": prec}
    if kind == "gemm":
        A, B = _factors(case, g)
        st.update(A=A, B=B, C=zb.empty_colmajor(case["m"], case["n"]), ta=bool(case["ta"]),
                  tb=bool(case["tb"]), slices=SLICES[case["prec"]])
    elif kind == "batch":
        members = _members(case)
        st["As"] = [_matrix(n, n, kappa, g) for n, kappa, _ in members]
        st["opts"] = [zb.opts(beta=1.0 / (kappa * guard), ns_steps=case["ns"], prec=prec)
                      for _, kappa, guard in members]
        # one buffer holds every Q_p, one every H; the call gets views of them
        total = sum(n * n for n, _, _ in members)
        st["Q"] = torch.empty(total, dtype=torch.float64, device="cuda")
        st["H"] = torch.empty(total, dtype=torch.float64, device="cuda")
        st["Qs"], st["Hs"], at = [], [], 0
        for n, _, _ in members:
            st["Qs"].append(st["Q"][at:at + n * n].view(n, n).t())
            st["Hs"].append(st["H"][at:at + n * n].view(n, n).t())
            at += n * n
    else:
        m, n = case["m"], case["n"]
        st["A"] = _matrix(m, n, case["kappa"], g)
        auto = case.get("auto", 0)
        st["o"] = zb.opts(beta=0.0 if auto else 1.0 / (case["kappa"] * case["guard"]),
                          alpha=0.0 if auto else 1.0, r=case["r"], ns_steps=case.get("ns", 0),
                          prec=prec)
        if kind == "pd":
            st["Qp"], st["Hm"] = zb.empty_colmajor(m, n), zb.empty_colmajor(n, n)
    return st


def _flip(U, V):
    """The sign of each singular vector pair made definite: the entry of u_i of
    largest magnitude is positive (a program that stores or compares vectors
    does this; the factorisation leaves it open)."""
    s = torch.sign(torch.gather(U, 0, U.abs().argmax(0, keepdim=True)))
    return U * s, V * s


def run(state):
    kind = state["kind"]
    if kind == "gemm":
        return zb.zolo_dgemm(state["h"], state["A"], state["B"], state["C"], transA=state["ta"],
                             transB=state["tb"], prec=state["prec"], slices=state["slices"])
    if kind == "pd":
        Qp, H, _ = zb.zolo_pd(state["h"], state["A"], state["o"], state["Qp"], state["Hm"])
        return {"Qp": Qp, "H": H}
    if kind == "batch":
        zb.zolo_pd_batched(state["h"], state["As"], state["opts"], state["Qs"], state["Hs"])
        return {"Qp": state["Q"], "H": state["H"]}
    U, S, V, _ = zb.zolo_svd(state["h"], state["A"], state["o"])
    U, V = _flip(U, V)
    return {"U": U, "S": S, "V": V}


# ------------------------------------------------------------------ the work
def _pd_flops(m, n, ell0, r, ns):
    """The Zolo-PD model: 5 r m n^2 per QR-form iteration, m n^2 + r (n^3 / 3 +
    2 m n^2) per Cholesky-form one, 4 m n^2 per Newton-Schulz step, 2 m n^2 for H."""
    _, qr, r = zb.schedule(min(1.0, ell0), r, 6)
    m, n = float(m), float(n)
    f = 2 * m * n * n + ns * 4 * m * n * n
    for q in qr:
        f += 5 * r * m * n * n if q else m * n * n + r * (n ** 3 / 3 + 2 * m * n * n)
    return f


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n), "flops": 2.0 * m * n * k}
    if kind == "batch":
        ms = _members(case)
        return {"bytes": sum(24.0 * n * n for n, _, _ in ms),
                "flops": sum(_pd_flops(n, n, 1.0 / (k * g), 0, case["ns"]) for n, k, g in ms)}
    m, n = case["m"], case["n"]
    if kind == "pd":
        # with bounds from the library, l_0 is near 1 / (sqrt(n) kappa) and a QR factor is formed
        ell0 = 1.0 / (case["kappa"] * case["guard"] * (math.sqrt(n) if case["auto"] else 1.0))
        f = _pd_flops(m, n, ell0, case["r"], case["ns"])
        return {"bytes": 8.0 * (2 * m * n + n * n),
                "flops": f + (2.0 * m * n * n if case["auto"] else 0.0)}
    # the eigendecomposition of H at the 9 n^3 of a tridiagonal method, U = Q_p V
    f = _pd_flops(m, n, 1.0 / (case["kappa"] * case["guard"]), case["r"], 0)
    return {"bytes": 8.0 * (2 * m * n + n * n + n),
            "flops": f + 9.0 * float(n) ** 3 + 2.0 * m * n * n}


# ------------------------------------------------------- the same in plain torch
def _polar(A):
    """A = Q_p H by the scaled Newton iteration on the triangular factor."""
    Q, X = torch.linalg.qr(A)
    R = X
    n = X.shape[0]
    for _ in range(14):
        Y = torch.linalg.inv(X).t()
        z = (torch.linalg.matrix_norm(Y, 1) * torch.linalg.matrix_norm(Y, math.inf)
             / (torch.linalg.matrix_norm(X, 1) * torch.linalg.matrix_norm(X, math.inf))) ** 0.25
        z = torch.where((z - 1).abs() < 1e-2, torch.ones_like(z), z)
        Xn = 0.5 * (z * X + Y / z)
        done = torch.linalg.matrix_norm(Xn - X) < 1e-9 * math.sqrt(n)
        X = Xn
        if bool(done):
            break
    X = 1.5 * X - 0.5 * X @ (X.t() @ X)
    H = X.t() @ R
    return Q @ X, 0.5 * (H + H.t())


def exact(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "gemm":
        A, B = _factors(case, g)
        return (A.t() if case["ta"] else A) @ (B.t() if case["tb"] else B)
    if kind == "pd":
        Qp, H = _polar(_matrix(case["m"], case["n"], case["kappa"], g))
        return {"Qp": Qp, "H": H}
    if kind == "batch":
        Qs, Hs = [], []
        for n, kappa, _ in _members(case):
            Qp, H = _polar(_matrix(n, n, kappa, g))
            Qs.append(Qp.t().reshape(-1))
            Hs.append(H.t().reshape(-1))
        return {"Qp": torch.cat(Qs), "H": torch.cat(Hs)}
    U, S, Vh = torch.linalg.svd(_matrix(case["m"], case["n"], case["kappa"], g).cpu(),
                                full_matrices=False)
    U, V = _flip(U, Vh.t())
    return {"U": U, "S": S, "V": V}
