"""Performance cases of libctm: what is timed, on which inputs, and what it computes.

Four groups, all through the public binding (paper_2112_13184_gb300.ctm):

* a scan point: one warm CTMRG sweep, the convergence measure and the reduced
  density matrices its observables come from (how a field or coupling scan
  advances), from the smallest cell in use to the S=1, D=8, chi=128 workload;
* several uneven instances advanced together (ctm_batch_sweep);
* observables alone: every one- and two-site density matrix, and correlation
  functions;
* single kernels at the shapes a sweep gives them: emulated-FP64 products,
  Householder QR, Jacobi SVD.

Handle-level passes return density matrices and correlations, which do not
depend on the basis of the chi bonds; the environment tensors do (their basis
is fixed only up to the projectors' gauge).  Site tensors are the package's
seeded product states plus noise; the environment starts from the product
boundary (only index 0 of every bond occupied), the usual start without an
earlier environment, and a few sweeps in prepare() bring it near its fixed
point, as in a scan.  The emulated-FP64 points cut singular values at 1e-8,
above what their products resolve, so that rounding is not carried into the
projectors; the FP64 points keep the default 1e-12.
"""
import math

import numpy as np
import torch

from paper_2112_13184_gb300 import ctm as C
from paper_2112_13184_gb300 import inputs as I

SETTLE = 3  # sweeps from the product boundary in prepare()


def _point(name, state, D, chi, precision, noise=0.05, bonds=8, sites=4):
    return dict(name=name, kind="point", state=state, D=D, chi=chi, precision=precision, noise=noise, bonds=bonds,
                sites=sites)


def listed():
    return [
        # smallest cell the parity runs use (N = chi D^2 = 32): every launch counts
        _point("point_fp64_d3_D2_chi8", "neel3", 2, 8, "fp64", 0.1),
        # the S=1/2 Heisenberg parity workload, exact projectors (N = 144)
        _point("point_fp64_d2_D3_chi16", "neel", 3, 16, "fp64", 0.1),
        # the smallest size of the serving family, emulated FP64
        _point("point_emu_d2_D4_chi32", "xpol", 4, 32, "emu"),
        # the FP64 arm at a middle size
        _point("point_fp64_d2_D6_chi48", "neel", 6, 48, "fp64"),
        # the headline workload (S=1, N = 8192), emulated FP64; energies on one bond of each direction
        _point("point_emu_d3_D8_chi128", "xpol3", 8, 128, "emu", 0.02, 2, 0),
        # uneven instances of a coupling scan advanced together, magnetisation of each
        dict(name="batch_emu_uneven", kind="batch", state="neel", sizes="3x24,4x32,5x32,6x48,4x64", precision="emu",
             noise=0.05),
        # all observables of one D=8 environment: 4 one-site and 8 two-site density matrices
        dict(name="measure_emu_d3_D8_chi64", kind="measure", state="xpol3", D=8, chi=64, precision="emu", noise=0.02,
             bonds=8, sites=4),
        # correlation functions along both axes from every site of the cell
        dict(name="corr_emu_d2_D5_chi48", kind="corr", state="xpol", D=5, chi=48, precision="emu", noise=0.05, rmax=6),
        # a range-finder apply of an enlarged corner (E^T X at N = 8192, k = 144)
        dict(name="gemm_emu_apply_8192x144", kind="gemm", M=8192, N=144, K=8192, tA=1, tB=0, slices=5),
        # the X3 product of an enlarged corner (short K, tall): chi = 64, D = 8, d = 3
        dict(name="gemm_emu_corner_262144x192", kind="gemm", M=262144, N=192, K=64, tA=0, tB=0, slices=5),
        # the range finder's basis at N = 8192, k = 144
        dict(name="qr_8192x144", kind="qr", N=8192, k=144),
        # the small factor's SVD in a warm sweep at chi = 128
        dict(name="svd_144", kind="svd", k=144, coupling=0.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("point", "point", "point", "batch", "measure", "corr", "gemm", "gemm", "qr", "svd"))
    if kind in ("point", "measure", "corr"):
        precision = rng.choice(("fp64", "emu"))
        D = rng.choice((2, 3, 4, 5, 6) if precision == "fp64" else (3, 4, 5, 6, 8))
        chi = _log(rng, max(8, 2 * D), {2: 40, 3: 40, 4: 56, 5: 48, 6: 48, 8: 64}[D])
        state = rng.choice(("neel", "xpol", "boson", "neel3", "xpol3"))
        noise = {2: 0.1, 6: 0.03, 8: 0.02}.get(D, 0.05)
        c = dict(kind=kind, state=state, D=D, chi=chi, precision=precision, noise=noise)
        if kind == "corr":
            return dict(c, rmax=rng.choice((1, 2, 3, 5, 8)))
        return dict(c, bonds=rng.choice((1, 2, 8)), sites=rng.choice((1, 4)))
    if kind == "batch":
        n = rng.randint(2, 6)
        sizes = ",".join("%dx%d" % (rng.choice((3, 4, 5, 6)), _log(rng, 20, 64)) for _ in range(n))
        return dict(kind="batch", state=rng.choice(("neel", "xpol")), sizes=sizes, precision="emu", noise=0.03)
    if kind == "gemm":
        tA, tB = rng.randint(0, 1), rng.randint(0, 1)
        if rng.random() < 0.5:  # applies: a square corner times a block of vectors
            n = _log(rng, 100, 7000)
            return dict(kind="gemm", M=n, N=_log(rng, 16, 144), K=n, tA=tA, tB=tB, slices=5)
        D = rng.choice((3, 4, 5, 6, 8))  # short-K corner products
        return dict(kind="gemm", M=_log(rng, 2000, 200000), N=D * D * rng.choice((1, 2, 3)), K=D * D * rng.choice((1, 2)),
                    tA=tA, tB=tB, slices=rng.choice((4, 5, 6)))
    if kind == "qr":
        k = _log(rng, 12, 160)
        return dict(kind="qr", N=_log(rng, max(64, k), 8192), k=k)
    return dict(kind="svd", k=_log(rng, 16, 160), coupling=rng.choice((0.02, 0.05, 0.1)))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
STATES = {
    "neel": (2, lambda D, a, s: I.neel_tensors(2, D, a, s), lambda: I.spin_ops(2)["Sz"]),
    "neel3": (3, lambda D, a, s: I.neel_tensors(3, D, a, s), lambda: I.spin_ops(3)["Sz"]),
    "xpol": (2, lambda D, a, s: I.x_polarised_tensors(2, D, a, s), lambda: I.spin_ops(2)["Sx"]),
    "xpol3": (3, lambda D, a, s: I.x_polarised_tensors(3, D, a, s), lambda: I.spin_ops(3)["Sx"]),
    "boson": (3, lambda D, a, s: I.uniform_boson_tensors(2, D, a, s), lambda: I.boson_ops(2)["n"]),
}


def _boundary(chi, D):
    """The product boundary: index 0 of every bond occupied."""
    e = {}
    for name, shape in I.env_shapes(chi, D).items():
        t = np.zeros(shape)
        t.flat[0] = 1.0
        e[name] = t
    return [e] * 4


def _handle(case, D, chi, seed):
    d, tensors, _ = STATES[case["state"]]
    emu = case["precision"] == "emu"
    c = C.CTMRG(d, D, chi, precision=C.CTM_OZAKI_BF16 if emu else C.CTM_FP64, sv_cutoff_rel=1e-8 if emu else 1e-12)
    c.set_tensors(tensors(D, case["noise"], seed))
    c.set_envs(_boundary(chi, D))
    c.sweep(SETTLE)
    return c


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gemm_inputs(case, seed):
    """Operands graded over their rows / columns as corners and bases are."""
    g = _gen(seed)
    M, N, K = case["M"], case["N"], case["K"]
    A = torch.randn((M, K), dtype=torch.float64, device="cuda", generator=g)
    A *= torch.logspace(0, -6, M, dtype=torch.float64, device="cuda")[:, None]
    B = torch.randn((K, N), dtype=torch.float64, device="cuda", generator=g)
    B *= torch.logspace(0, -6, N, dtype=torch.float64, device="cuda")[None, :]
    return (A.t().contiguous() if case["tA"] else A), (B.t().contiguous() if case["tB"] else B)


def _qr_input(case, seed):
    """Columns graded over 12 decades, as a warm range finder gives them."""
    Y = torch.randn((case["N"], case["k"]), dtype=torch.float64, device="cuda", generator=_gen(seed))
    return Y * torch.logspace(0, -12, case["k"], dtype=torch.float64, device="cuda")[None, :]


def _svd_input(case, seed):
    """R^T of a warm cut: lower triangular, graded rows, weakly coupled."""
    k = case["k"]
    s = torch.logspace(0, -12, k, dtype=torch.float64, device="cuda")
    L = case["coupling"] * torch.randn((k, k), dtype=torch.float64, device="cuda", generator=_gen(seed))
    return ((torch.tril(L, -1) + torch.eye(k, dtype=torch.float64, device="cuda")) * s[:, None]).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind in ("point", "measure", "corr"):
        st["h"] = _handle(case, case["D"], case["chi"], seed)
    elif kind == "batch":
        st["hs"] = [_handle(case, D, chi, seed + 1000 * j) for j, (D, chi) in enumerate(_sizes(case))]
    elif kind == "gemm":
        st["A"], st["B"] = _gemm_inputs(case, seed)
        M, N, K = case["M"], case["N"], case["K"]
        st["C"] = torch.empty((M, N), **f64)
        st["ws"] = torch.zeros(C.ctm_gemm_ozaki_workspace_bytes(M, N, K, case["slices"]), dtype=torch.uint8, device="cuda")
    elif kind == "qr":
        N, k = case["N"], case["k"]
        st["Y"] = _qr_input(case, seed)
        st["Q"], st["R"] = torch.empty((N, k), **f64), torch.empty((k, k), **f64)
        st["ws"] = torch.empty(C.ctm_qr_workspace_bytes(N, k), dtype=torch.uint8, device="cuda")
    else:
        k = case["k"]
        st["G"] = _svd_input(case, seed)
        st["U"], st["S"], st["V"] = torch.empty((k, k), **f64), torch.empty(k, **f64), torch.empty((k, k), **f64)
        st["ws"] = torch.empty(C.ctm_svd_workspace_bytes(k), dtype=torch.uint8, device="cuda")
    return st


def _measure(c, sites, bonds):
    out = {"rho1": [c.rdm1(i) for i in range(sites)]}
    out["rho2"] = [c.rdm2(i, dx, dy) for i, dx, dy in I.SQUARE_2X2_BONDS[:bonds]]
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "point":
        c = state["h"]
        c.sweep(1)
        c.loop_delta()
        return _measure(c, case["sites"], case["bonds"])
    if kind == "measure":
        return _measure(state["h"], case["sites"], case["bonds"])
    if kind == "corr":
        op = STATES[case["state"]][2]()
        return state["h"].correlation(op, op, case["rmax"])
    if kind == "batch":
        C.ctm_batch_sweep([c.h for c in state["hs"]], 1)
        return [[c.rdm1(i) for i in range(4)] for c in state["hs"]]
    if kind == "gemm":
        A, B = state["A"], state["B"]
        C.ctm_gemm_ozaki(case["tA"], case["tB"], case["M"], case["N"], case["K"], 1.0, A, A.shape[1], B, B.shape[1],
                         0.0, state["C"], case["N"], case["slices"], state["ws"])
        return state["C"]
    if kind == "qr":
        C.ctm_qr(state["Y"], case["N"], case["k"], state["Q"], state["R"], state["ws"])
        return state["Q"], state["R"]
    C.ctm_svd(state["G"], case["k"], state["U"], state["S"], state["V"], state["ws"])
    return state["U"], state["S"], state["V"]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _corner_flops(d, D, chi):
    """One enlarged corner: C T, then the edge, the ket and the bra."""
    N = chi * D * D
    return 2.0 * chi * chi * N + 2.0 * N * N * chi + 4.0 * N * N * d * D * D


def _sweep_flops(d, D, chi):
    """One warm sweep: per cut four corners, a subspace iteration (eight
    products with a corner), two QRs, the small factor's SVD, four products
    for the projectors, and the absorption of one site."""
    N = chi * D * D
    k = N if N <= 256 else min(N, chi + max(8, chi // 8))
    cut = 4 * _corner_flops(d, D, chi) + 8 * 2.0 * N * N * k + 2 * 4.0 * N * k * k + 8.0 * k ** 3
    cut += 4 * 2.0 * N * N * chi + 4.0 * N * k * chi
    absorb = _corner_flops(d, D, chi) + 2.0 * N * N * chi + 6.0 * N * chi * chi
    return 16 * (cut + absorb)


def _state_bytes(d, D, chi):
    return 8.0 * (4 * d * D ** 4 + 16 * chi * chi + 16 * chi * chi * D * D)


def _rdm1_flops(d, D, chi):
    """The corner with both physical legs open, and the ring around it."""
    N = chi * D * D
    return 2.0 * N * N * chi + 2.0 * N * N * d * D * D + 2.0 * N * N * d * d * D * D + 4.0 * N * N * chi + 2.0 * N * N * d * d


def _rdm2_flops(d, D, chi):
    """Two open halves, each closed with an edge and a corner."""
    N = chi * D * D
    half = 2.0 * N * N * chi + 2.0 * N * N * d * D * D + 2.0 * N * N * d * d * D * D + 2.0 * N * d * d * N * chi
    return 2 * half + 2.0 * d ** 4 * N * chi


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + K * N + M * N), "flops": 2.0 * M * N * K}
    if kind == "qr":
        N, k = case["N"], case["k"]
        return {"bytes": 8.0 * (2 * N * k + k * k), "flops": 4.0 * N * k * k}
    if kind == "svd":
        k = case["k"]
        return {"bytes": 8.0 * (3 * k * k + k), "flops": 20.0 * k ** 3}
    d = STATES[case["state"]][0]
    if kind == "batch":
        s = _sizes(case)
        return {"bytes": sum(2 * _state_bytes(d, D, chi) for D, chi in s),
                "flops": sum(_sweep_flops(d, D, chi) + 4 * _rdm1_flops(d, D, chi) for D, chi in s)}
    D, chi = case["D"], case["chi"]
    if kind == "corr":
        columns = 2 * 4 * (3 * case["rmax"] + 2)
        N = chi * D * D
        return {"bytes": _state_bytes(d, D, chi), "flops": columns * (_corner_flops(d, D, chi) + 2.0 * N * N * chi)}
    flops = case["sites"] * _rdm1_flops(d, D, chi) + case["bonds"] * _rdm2_flops(d, D, chi)
    if kind == "measure":
        return {"bytes": _state_bytes(d, D, chi), "flops": flops}
    return {"bytes": 2 * _state_bytes(d, D, chi), "flops": flops + _sweep_flops(d, D, chi)}


# --------------------------------------------------------------------------
# the same in plain 64-bit torch / numpy
# --------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B = _gemm_inputs(case, seed)
        return (A.t() if case["tA"] else A) @ (B.t() if case["tB"] else B)
    if kind == "qr":
        Q, R = np.linalg.qr(_qr_input(case, seed).cpu().numpy())
        s = np.where(np.diag(R) < 0, -1.0, 1.0)
        return Q * s[None, :], R * s[:, None]
    if kind == "svd":
        # the signs of the singular vectors are free
        return None, np.linalg.svd(_svd_input(case, seed).cpu().numpy(), compute_uv=False), None
    return None
