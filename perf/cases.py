"""The work that the ladder library is asked to do, case by case, through its public entry points.

Each case is a plain dict; `prepare` makes what a coupled-cluster program has in hand before the
call (Cholesky vectors, amplitudes, the output array and the workspace that it keeps over its
iterations), `run` makes the one call, `exact` gives the same result in 64 bits by plain torch.

kind  fwd   ladder_forward: one evaluation of the ladder term (and of the pair energy)
      grad  ladder() and its backward through autograd: value, dL and dt2
      bwd   ladder_backward: the adjoint alone, dL and dt2
      term  tijkl / tijbk: the two further Cholesky terms of the vector function
sym   t2[i,j,a,b] = t2[j,i,b,a], the closed-shell case, is promised to the library
"""
import math

import torch

from paper_2310_04559_gb300 import binding as B
from paper_2310_04559_gb300 import synth

GIB = 1 << 30
LARGEST = 2.0 * (40 * 40 + 2000) * 400.0 ** 4  # multiply-adds (x 2) of the largest listed case


def listed():
    return [
        # the smallest evaluation there is, FP64, with the energy: a test molecule, all launches and latency
        dict(name="fp64_tiny", kind="fwd", o=4, v=24, n=60, mode="fp64", sym=True, energy=True, budget_gib=1),
        # the same size as a differentiable layer, value and both gradients: orbital relaxation of a small molecule
        dict(name="grad_tiny", kind="grad", o=4, v=24, n=60, mode="ozaki_bf16", sym=True),
        # few occupied orbitals (v >> o): the planner is free to take the Cholesky-first order
        dict(name="fwd_few_occupied", kind="fwd", o=4, v=96, n=480, mode="ozaki_bf16", sym=True, energy=False, budget_gib=8),
        # amplitudes without pair symmetry (response and Lambda equations), odd sizes
        dict(name="fwd_general_odd", kind="fwd", o=11, v=137, n=613, mode="ozaki_bf16", sym=False, energy=False, budget_gib=16),
        # an everyday CCSD iteration, ladder term and pair energy
        dict(name="fwd_ordinary", kind="fwd", o=20, v=200, n=1000, mode="ozaki_bf16", sym=True, energy=True, budget_gib=32),
        # the benchmark's workload, in a device that the rest of the CC program shares
        dict(name="fwd_large", kind="fwd", o=40, v=400, n=2000, mode="ozaki_bf16", sym=True, energy=True, budget_gib=48),
        # early iterations in BF16, odd sizes
        dict(name="fwd_bf16_odd", kind="fwd", o=27, v=301, n=1501, mode="bf16", sym=True, energy=False, budget_gib=48),
        # early iterations in TF32, the everyday size
        dict(name="fwd_tf32", kind="fwd", o=20, v=200, n=1000, mode="tf32", sym=True, energy=False, budget_gib=32),
        # the reference precision, for validating a calculation
        dict(name="fwd_fp64", kind="fwd", o=10, v=100, n=500, mode="fp64", sym=True, energy=True, budget_gib=8),
        # the adjoint of the stated workload
        dict(name="bwd_adjoint", kind="bwd", o=16, v=160, n=800, mode="ozaki_bf16", sym=True, budget_gib=32),
        # Eq. 9 of the vector function, beside the ladder in every iteration
        dict(name="term_ijbk", kind="term", which="ijbk", o=20, v=200, n=1000, mode="ozaki_bf16", budget_gib=32),
        # amplitudes that outgrow the device: t2 and R stay in page-locked host memory
        dict(name="fwd_host_amplitudes", kind="fwd", o=30, v=150, n=750, mode="ozaki_bf16", sym=True, energy=False, host_t2r=True, budget_gib=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the listed ranges (o << v << n, n about 4 to 6 times o + v)."""
    kind = rng.choice(["fwd", "fwd", "fwd", "fwd", "grad", "bwd", "term"])
    mode = rng.choice(["ozaki_bf16", "ozaki_bf16", "ozaki_bf16", "fp64", "tf32", "bf16"]) if kind == "fwd" else "ozaki_bf16"
    vmax = {"fp64": 110, "tf32": 301, "bf16": 301}.get(mode, 400)
    vmax = {"grad": 96, "bwd": 180, "term": 240}.get(kind, vmax)
    while True:
        v = _log(rng, 24, vmax)
        o = max(2, int(round(v * rng.uniform(0.04, 0.17))))
        n = max(8, int(round((o + v) * rng.uniform(4.0, 5.5))))
        if 2.0 * (o * o + n) * float(v) ** 4 <= LARGEST:
            break
    case = dict(kind=kind, o=o, v=v, n=n, mode=mode)
    if kind == "fwd":
        case["sym"] = rng.random() < 0.7 or v > 200
        case["energy"] = rng.random() < 0.5
        case["budget_gib"] = 48 if v > 200 else 32
        if case["sym"] and mode == "ozaki_bf16" and not case["energy"] and v <= 160:
            case["host_t2r"] = rng.random() < 0.4
    elif kind == "grad":
        case["sym"] = rng.random() < 0.5
    elif kind == "bwd":
        case["sym"] = rng.random() < 0.5
        case["budget_gib"] = 32
    else:
        case["which"] = rng.choice(["ijkl", "ijbk"])
        case["budget_gib"] = 32
    return case


def _inputs(case, seed):
    """L, t2 and, where the case has them, W and Lov: the seeded recipe of the package on the device."""
    o, v, n = case["o"], case["v"], case["n"]
    L, t2 = synth.ladder_inputs_torch(o, v, n, seed=seed, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed + 7919)
    x = {"L": L, "t2": t2}
    if not case.get("sym", False):
        t2.copy_(torch.randn(t2.shape, generator=g, dtype=torch.float64, device="cuda").mul_(1e-2))
    if case["kind"] in ("grad", "bwd"):
        x["W"] = torch.randn(t2.shape, generator=g, dtype=torch.float64, device="cuda")
    if case["kind"] == "term":
        Lov = torch.randn((n, o, v), generator=g, dtype=torch.float64, device="cuda")
        x["Lov"] = Lov * torch.exp(-5.0 * torch.arange(n, dtype=torch.float64, device="cuda") / n)[:, None, None]
    return x


def prepare(case, seed):
    o, v, n, kind = case["o"], case["v"], case["n"], case["kind"]
    s = dict(_inputs(case, seed), case=dict(case))
    budget = case.get("budget_gib", 0) * GIB
    if kind == "fwd":
        host = bool(case.get("host_t2r", False))
        kw = dict(mode=case["mode"], symmetric=case["sym"], budget=budget, host_t2r=host)
        if host:
            pinned = torch.empty(s["t2"].shape, dtype=torch.float64, pin_memory=True)
            pinned.copy_(s["t2"])
            s["t2"] = pinned
            s["R"] = torch.empty(pinned.shape, dtype=torch.float64, pin_memory=True)
        else:
            s["R"] = torch.empty_like(s["t2"])
        s["ws"] = B.alloc_workspace(B.workspace_size(o, v, n, **kw), s["L"].device)
        s["kw"] = dict(kw, energy=case["energy"])
    elif kind == "grad":
        s["L"].requires_grad_()
        s["t2"].requires_grad_()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fwd":
        return B.ladder_forward(s["L"], s["t2"], R=s["R"], workspace=s["ws"], **s["kw"])
    if kind == "grad":
        R = B.ladder(s["L"], s["t2"], mode=case["mode"], symmetric=case["sym"])
        dL, dt2 = torch.autograd.grad(R, (s["L"], s["t2"]), s["W"])
        return R.detach(), dL, dt2
    if kind == "bwd":
        return B.ladder_backward(s["L"], s["t2"], s["W"], mode=case["mode"], symmetric=case["sym"],
                                 budget=case["budget_gib"] * GIB)
    if case["which"] == "ijkl":
        return B.tijkl(s["Lov"], s["t2"], mode=case["mode"], budget=case["budget_gib"] * GIB)
    return B.tijbk(s["Lov"], s["L"], s["t2"], mode=case["mode"], budget=case["budget_gib"] * GIB)


def _ladder_flops(o, v, n, sym):
    """The fewest flops known for one evaluation: integrals for b >= a only, the ladder on the parts
    symmetric and antisymmetric in c, d, or the Cholesky-first order where that is less."""
    vv = float(v) * v
    pp, pm = (o * (o + 1) / 2, o * (o - 1) / 2) if sym else (o * o, o * o)
    packed = vv * (n * float(v) * (v + 1) + 2.0 * (pp * v * (v + 1) / 2 + pm * v * (v - 1) / 2))
    return min(packed, 4.0 * n * pp * float(v) ** 3)


def work(case):
    o, v, n, kind = case["o"], case["v"], case["n"], case["kind"]
    amp, chol = 8.0 * o * o * v * v, 8.0 * n * v * v
    sym = case.get("sym", False)
    if kind == "fwd":
        return {"bytes": chol + 2 * amp, "flops": _ladder_flops(o, v, n, sym)}
    # the adjoint: one evaluation with the cotangent (no pair symmetry) for dt2; for dL the block
    # sum_ij W_ijeb t_ijfd and its contraction with L, once (sym) or twice
    back = _ladder_flops(o, v, n, False) + (1 if sym else 2) * 2.0 * (o * o + n) * float(v) ** 4
    if kind == "bwd":
        return {"bytes": 2 * chol + 3 * amp, "flops": back}
    if kind == "grad":
        return {"bytes": 2 * chol + 4 * amp, "flops": _ladder_flops(o, v, n, sym) + back}
    q = o if case["which"] == "ijkl" else v
    return {"bytes": 8.0 * n * o * v + (chol if q == v else 0) + amp + 8.0 * o * o * o * q,
            "flops": 2.0 * (n + o * o) * o * q * float(v) * v}


def _general(A, Bm, t2):
    """G[i,j,p,q] = sum_cd (sum_P A[P,p,c] B[P,q,d]) t2[i,j,c,d], one p at a time."""
    o, v = t2.shape[0], t2.shape[2]
    n, np_, nq = A.shape[0], A.shape[1], Bm.shape[1]
    t = t2.reshape(o * o, v * v)
    Bf = Bm.reshape(n, nq * v)
    G = torch.empty((o * o, np_, nq), dtype=torch.float64, device=t2.device)
    for p in range(np_):
        V = (A[:, p, :].t().contiguous() @ Bf).reshape(v, nq, v)
        G[:, p, :] = t @ V.permute(1, 0, 2).reshape(nq, v * v).t()
    return G.reshape(o, o, np_, nq)


def _energy(R, t2):
    return ((2.0 * R - R.transpose(2, 3)) * t2).sum()


def _adjoint(L, t2, W):
    o, v, n = t2.shape[0], t2.shape[2], L.shape[0]
    LT = L.transpose(1, 2).contiguous()
    dt2 = _general(LT, LT, W)
    # R_ijab = sum L_Pac L_Pbd t_ijcd: both places of L
    dL = torch.zeros_like(L)
    Lf = L.reshape(n, v * v)
    for X, t in ((W, t2), (W.permute(1, 0, 3, 2), t2.permute(1, 0, 3, 2))):
        Xf, tf = X.reshape(o * o, v, v), t.reshape(o * o, v * v)
        for a in range(v):
            M = (Xf[:, a, :].t() @ tf).reshape(v, v, v)  # [b, c, d]
            dL[:, a, :] += Lf @ M.permute(1, 0, 2).reshape(v, v * v).t()
    return dL, dt2


def exact(case, seed):
    o, v, n, kind = case["o"], case["v"], case["n"], case["kind"]
    flops = 2.0 * (o * o + n) * float(v) ** 4 * {"fwd": 1, "grad": 4, "bwd": 3}.get(kind, float(o) / v)
    if flops > 8e12:  # over about 20 seconds of FP64
        return None
    x = _inputs(case, seed)
    if kind == "fwd":
        R = _general(x["L"], x["L"], x["t2"])
        E = _energy(R, x["t2"])
        if case.get("host_t2r", False):
            R = R.cpu()
        return (R, E) if case["energy"] else R
    if kind == "term":
        if case["which"] == "ijkl":
            return _general(x["Lov"], x["Lov"], x["t2"])
        return _general(x["Lov"], x["L"], x["t2"]).transpose(2, 3).contiguous()
    dL, dt2 = _adjoint(x["L"], x["t2"], x["W"])
    if kind == "bwd":
        return dL, dt2
    return _general(x["L"], x["L"], x["t2"]), dL, dt2
