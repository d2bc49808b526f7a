"""The work whose speed is tracked: what a program that computes disconnected
twisted-mass loops calls, through the public entry points, from a 4^4 test
lattice to the 32^3 x 64 workload.

Kinds of cases (``kind``):
  dslash   one application of the operator (M, M^dag, D_W, gamma_5 D_W, or a
           fourth-order hopping expansion) to n systems, in any precision;
  solve    one batched CG call (plain or mixed precision);
  group    several lattices of unlike size solved in one call;
  loops    the loop contractions of n solutions with both one-end estimators;
  momenta  momentum-projected local loops;
  tsm      a whole Truncated Solver Method estimate (noise to combined loops).

Inputs come from the case's seed alone: links U = exp(0.3 i H) with Gaussian
traceless Hermitian H, the fields complex Gaussian (the operator and the
contractions meet CG vectors and solutions, which look like that) or the Z4
sources that solves start from.  ``exact`` evaluates the same path in
complex128 with plain torch.
"""
import math

import torch

from paper_1401_6749_gb300 import tmloops as tl
from paper_1401_6749_gb300.tsm_pipeline import TsmPipeline

C128 = torch.complex128

# what the paper's observables need: the sigma terms (one-end trick), g_A and
# the one-derivative operator (generalised one)
TSM_KINDS = ("local_vv", "local_gen", "oneD_gen")


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the operator alone on the production lattice: one FP32 system, the
        # figure that Dslash implementations are quoted by
        dict(name="dslash-32x64-f32-1", kind="dslash", X=32, Y=32, Z=32, T=64, n=1, prec="f32", layout="std",
             op="M", recon=0),
        # the truncated solves' operator: 16 FP16 systems in the interleaved
        # layout, also applied by itself for the generalised estimator
        dict(name="dslash-32x64-il-f16-16", kind="dslash", X=32, Y=32, Z=32, T=64, n=16, prec="f16", layout="il",
             op="DW", recon=0),
        # the FP64 operator a program checks its solutions with, small lattice
        dict(name="dslash-16x32-f64-1", kind="dslash", X=16, Y=16, Z=16, T=32, n=1, prec="f64", layout="std",
             op="M", recon=0),
        # the smallest work: plain FP64 CG of 16 sources on 4^4 to 1e-10
        dict(name="solve-4x4-f64-16", kind="solve", X=4, Y=4, Z=4, T=4, n=16, mode="plain", prec="f64", layout="std",
             tol=1e-10, kappa=0.16, mu=0.01, schur=False, graph=False, every=8, iters=56),
        # one source to high precision with FP64 reliable updates
        dict(name="solve-16x32-mixed-1", kind="solve", X=16, Y=16, Z=16, T=32, n=1, mode="mixed", prec="f32",
             layout="std", tol=1e-10, kappa=0.16, mu=0.005, schur=True, graph=False, every=4, iters=32),
        # a batch of high-precision solves, iterations replayed as a graph
        dict(name="solve-24x48-mixed-12", kind="solve", X=24, Y=24, Z=24, T=48, n=12, mode="mixed", prec="f32",
             layout="std", tol=1e-9, kappa=0.161, mu=0.004, schur=True, graph=True, every=4, iters=32),
        # one batch of truncated FP16 solves of the production workload
        dict(name="solve-32x64-il-f16-16", kind="solve", X=32, Y=32, Z=32, T=64, n=16, mode="plain", prec="f16",
             layout="il", tol=1e-2, kappa=0.161, mu=0.003, schur=True, graph=False, every=2, iters=6),
        # truncated solves of an uneven batch of lattices in one call
        dict(name="group-8-12-16-24", kind="group", sets="8.8.8.8:4,12.12.12.12:8,16.16.16.32:16,24.24.24.48:32",
             prec="f16", tol=1e-2, graph=True, every=2, iters=6),
        # the loops of one batch of truncated solutions: D_W, local and
        # one-derivative operators, both estimators
        dict(name="loops-32x64-il-f16-16", kind="loops", X=32, Y=32, Z=32, T=64, n=16, prec="f16", layout="il"),
        # the loops of high-precision solutions: FP64 solutions converted to
        # float-float, then the same operators
        dict(name="loops-24x48-ff-8", kind="loops", X=24, Y=24, Z=24, T=48, n=8, prec="ff", layout="std"),
        # local loops at the 19 momenta with n^2 <= 2
        dict(name="momenta-24x48-f32-12", kind="momenta", X=24, Y=24, Z=24, T=48, n=12, prec="f32", n2max=2),
        # a whole estimate: 60 truncated and 4 high-precision sources
        dict(name="tsm-16x32-60-4", kind="tsm", X=16, Y=16, Z=16, T=32, n_lp=60, n_hp=4, batch=16, prec="f16",
             kappa=0.161, mu=0.004),
    ]


def _extents(rng, vmin, vmax):
    """Even extents (X, Y, Z, T), rarely equal, with a volume spread over the logarithm of [vmin, vmax]."""
    while True:
        v = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
        side = (v / 2.0) ** 0.25  # T about twice the spatial extents
        L = [max(2, 2 * round(side * rng.uniform(0.7, 1.4) / 2)) for _ in range(3)]
        L.append(max(2, 2 * round(v / (L[0] * L[1] * L[2]) / 2)))
        if all(e >= 4 for e in L) and L[3] <= 96 and vmin <= L[0] * L[1] * L[2] * L[3] <= vmax:
            return L


def _systems(rng, L, most_sites, most):
    """1 to `most` systems, at most `most_sites` site-systems."""
    cap = max(1, min(most, most_sites // (L[0] * L[1] * L[2] * L[3])))
    return rng.randint(1, cap)


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "solve", "solve", "group", "loops", "momenta", "tsm"])
    full = 32 * 32 * 32 * 64
    dims = lambda L: dict(X=L[0], Y=L[1], Z=L[2], T=L[3])  # noqa: E731
    if kind == "dslash":
        prec, layout = rng.choice([("f32", "std"), ("f32", "std"), ("f64", "std"), ("ff", "std"), ("f16", "std"),
                                   ("f16", "il"), ("f16", "il"), ("bf16", "il")])
        wide = prec in ("f64", "ff")
        L = _extents(rng, 256, full // 4 if wide else full)
        n = _systems(rng, L, (full // 2) if wide else 16 * full if layout == "il" else 8 * full, 24)
        op = rng.choice(["M", "Mdag", "DW"] if layout == "il" else ["M", "Mdag", "DW", "g5DW", "hpe4"])
        recon = 0 if layout == "il" else rng.choice([0, 0, 12, 18])
        return dict(kind=kind, **dims(L), n=n, prec=prec, layout=layout, op=op, recon=recon)
    if kind == "solve":
        mode, prec, layout, tol = rng.choice([("plain", "f64", "std", 1e-10), ("plain", "f32", "std", 1e-5),
                                              ("mixed", "f32", "std", 1e-9), ("mixed", "f16", "std", 1e-9),
                                              ("plain", "f16", "il", 1e-2), ("plain", "bf16", "il", 1e-2),
                                              ("plain", "f16", "std", 1e-2)])
        low = prec in ("f16", "bf16") and mode == "plain"
        L = _extents(rng, 256, full if low else full // 8 if prec == "f64" else full // 4)
        n = _systems(rng, L, 16 * full if low else full // 8 if prec == "f64" else full, 24)
        schur = rng.random() < 0.7
        iters = (6 if low else 22 if prec == "f32" and mode == "plain" else 32) * (1 if schur else 3)
        return dict(kind=kind, **dims(L), n=n, mode=mode, prec=prec, layout=layout, tol=tol,
                    kappa=round(rng.uniform(0.155, 0.161), 4), mu=round(rng.uniform(0.003, 0.01), 4), schur=schur,
                    graph=rng.random() < 0.5, every=rng.choice([2, 4]), iters=iters)
    if kind == "group":
        sets = []
        for _ in range(rng.randint(2, 4)):
            L = _extents(rng, 2048, full // 4)
            sets.append("%d.%d.%d.%d:%d" % (*L, _systems(rng, L, 4 * full, 24)))
        return dict(kind=kind, sets=",".join(sets), prec=rng.choice(["f16", "bf16"]), tol=1e-2,
                    graph=rng.random() < 0.5, every=2, iters=6)
    if kind == "loops":
        prec, layout = rng.choice([("f16", "il"), ("bf16", "il"), ("ff", "std"), ("f64", "std"), ("f32", "std"),
                                   ("f16", "std")])
        wide = prec in ("f64", "ff")
        L = _extents(rng, 256, full // 4 if wide else full)
        n = _systems(rng, L, full if wide else 16 * full if layout == "il" else 4 * full, 20)
        return dict(kind=kind, **dims(L), n=n, prec=prec, layout=layout)
    if kind == "momenta":
        L = _extents(rng, 256, full // 4)
        return dict(kind=kind, **dims(L), n=_systems(rng, L, 2 * full, 16),
                    prec=rng.choice(["f16", "f32", "f64", "ff"]), n2max=rng.choice([0, 1, 2, 3]))
    L = _extents(rng, 256, 16 * 16 * 16 * 32)
    return dict(kind="tsm", **dims(L), n_lp=rng.randint(2, 60), n_hp=rng.randint(1, 4), batch=rng.choice([8, 16, 20]),
                prec=rng.choice(["f16", "bf16"]), kappa=0.16, mu=round(rng.uniform(0.003, 0.01), 4))


# ------------------------------------------------------------------ inputs
def _dims(c):
    return (c["X"], c["Y"], c["Z"], c["T"])


def _generator(seed, what):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + what)


def _gauge(L, seed):
    """exp(0.3 i H), H = sum_a w_a lambda_a / 2 with w_a ~ N(0, 1): complex128 (4, T, Z, Y, X, 3, 3)."""
    X, Y, Z, T = L
    gen = _generator(seed, 1)
    U = torch.empty((4, T, Z, Y, X, 3, 3), dtype=C128, device="cuda")
    s3 = 1.0 / math.sqrt(3.0)
    for mu in range(4):
        w = 0.15 * torch.randn((8, T, Z, Y, X), generator=gen, dtype=torch.float64, device="cuda")
        A = torch.zeros((3, 3, T, Z, Y, X), dtype=C128, device="cuda")  # i * 0.3 * H, matrix indices first
        for (i, j), (re, im) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
            A[i, j] = torch.complex(w[im], w[re])
            A[j, i] = torch.complex(-w[im], w[re])
        zero = torch.zeros_like(w[0])
        for i, d in enumerate((w[2] + s3 * w[7], -w[2] + s3 * w[7], -2 * s3 * w[7])):
            A[i, i] = torch.complex(zero, d)
        E = torch.zeros_like(A)
        for i in range(3):
            E[i, i] = 1
        for k in range(18, 0, -1):  # Horner form of the exponential series
            E = torch.stack([torch.stack([A[i, 0] * E[0, j] + A[i, 1] * E[1, j] + A[i, 2] * E[2, j]
                                          for j in range(3)]) for i in range(3)]) / k
            for i in range(3):
                E[i, i] += 1
        U[mu] = E.permute(2, 3, 4, 5, 0, 1)
    return U


def _spinors(L, n, seed, what=2):
    """Complex Gaussian spinors (n, T, Z, Y, X, 4, 3)."""
    X, Y, Z, T = L
    out = torch.empty((n, T, Z, Y, X, 4, 3), dtype=C128, device="cuda")
    return torch.view_as_real(out).normal_(generator=_generator(seed, what)).view(-1).view(C128).view(out.shape)


def _pack(L, psi, prec):
    f = tl.empty_field(L, prec, psi.shape[0])
    tl.tm_spinor_pack(L, f, prec, psi, psi.shape[0])
    return f


def _pack_layout(L, psi, prec, layout):
    f = _pack(L, psi, prec)
    if layout == "std":
        return f
    g = tl.empty_field_il(L, psi.shape[0])
    tl.tm_spinor_to_il(L, g, f, prec, psi.shape[0])
    return g


def _operator(case, U):
    return tl.Operator(_dims(case), case.get("kappa", 0.161), case.get("mu", 0.003), U, recon=case.get("recon", 0))


def _params(case):
    prec = tl.PREC[case["prec"]]
    if case.get("mode", "plain") == "mixed":
        return tl.cg_params(case["tol"], 2000, tl.CG_MIXED, inner_prec=prec, delta=0.1, check_every=case["every"],
                            schur=case["schur"], graph=case["graph"])
    return tl.cg_params(case["tol"], 2000, tl.CG_PLAIN, prec=prec, check_every=case["every"],
                        schur=case.get("schur", True), graph=case["graph"])


def _sets(case):
    """(L, n, kappa, mu) of each set of a group."""
    out = []
    for i, s in enumerate(case["sets"].split(",")):
        ext, n = s.split(":")
        out.append((tuple(int(e) for e in ext.split(".")), int(n), 0.155 + 0.002 * i, 0.01 - 0.002 * i))
    return out


def _momenta(case):
    k = range(-1, 2)
    return [(a, b, c) for a in k for b in k for c in k if a * a + b * b + c * c <= case["n2max"]]


_VIEW = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "ff": torch.float32}


def prepare(case, seed):
    kind, prec = case["kind"], tl.PREC[case["prec"]]
    st = dict(case=case, prec=prec)
    if kind == "group":
        st["ops"], st["eta"], st["x"], st["n"] = [], [], [], []
        for i, (L, n, kappa, mu) in enumerate(_sets(case)):
            st["ops"].append(tl.Operator(L, kappa, mu, _gauge(L, seed + 100 * i), recon=0))
            eta = tl.empty_field(L, prec, n)
            tl.z4_noise(L, eta, prec, seed + i, 0, n)
            st["eta"].append(eta)
            st["x"].append(tl.empty_field(L, prec, n))
            st["n"].append(n)
        st["params"] = _params(case)
        return st
    L = _dims(case)
    st["L"] = L
    if kind == "momenta":
        st["left"] = _pack(L, _spinors(L, case["n"], seed), prec)
        st["right"] = _pack(L, _spinors(L, case["n"], seed, 3), prec)
        st["out"] = torch.empty((case["n"], len(_momenta(case)), 16, L[3], 2), dtype=torch.float64, device="cuda")
        st["mom"] = _momenta(case)
        return st
    st["op"] = op = _operator(case, _gauge(L, seed))
    if kind == "tsm":
        st["pipe"] = TsmPipeline(op, case["n_hp"], case["n_lp"], batch=case["batch"], lp_prec=prec,
                                 hp_loop_prec=tl.FF, seed=seed, kinds=TSM_KINDS)
        return st
    n = case["n"]
    if kind == "dslash":
        st["in"] = _pack_layout(L, _spinors(L, n, seed), prec, case["layout"])
        st["out"] = torch.empty_like(st["in"])
    elif kind == "solve":
        st["params"] = _params(case)
        if case["layout"] == "il":
            st["eta"], st["x"] = tl.empty_field_il(L, n), tl.empty_field_il(L, n)
            tl.z4_noise_il(L, st["eta"], prec, seed, 0, n)
        else:
            hi = tl.F64 if case["mode"] == "mixed" else prec
            st["eta"], st["x"] = tl.empty_field(L, hi, n), tl.empty_field(L, hi, n)
            tl.z4_noise(L, st["eta"], hi, seed, 0, n)
    else:  # loops; float-float ones start from the FP64 solutions
        psi = _spinors(L, n, seed)
        if case["prec"] == "ff":
            st["x64"] = _pack(L, psi, tl.F64)
            st["x"] = torch.empty_like(st["x64"])
        else:
            st["x"] = _pack_layout(L, psi, prec, case["layout"])
        st["dw"] = torch.empty_like(st["x"])
        st["local"] = [torch.empty((n, 16, L[3], 2), dtype=torch.float64, device="cuda") for _ in range(2)]
        st["oned"] = [torch.empty((n, 4, 16, L[3], 2), dtype=torch.float64, device="cuda") for _ in range(2)]
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case, prec = st["case"], st["prec"]
    kind = case["kind"]
    if kind == "group":
        tl.tm_cg_solve_group(st["ops"], st["x"], st["eta"], st["n"], st["params"])
        return [x.view(_VIEW[case["prec"]]) for x in st["x"]]
    L = st["L"]
    if kind == "tsm":
        pipe = st["pipe"]
        res = pipe.run()
        out = {"est_" + k: [m, e] for k, (m, e) in res.items()}
        out.update({"lp_" + k: v for k, v in pipe.lp_loops.items()})
        out.update({"hp_" + k: v for k, v in pipe.hp_loops.items()})
        return out
    n = case["n"]
    if kind == "dslash":
        args = dict(dagger=case["op"] == "Mdag", mu_zero=case["op"] in ("DW", "g5DW"), prec=prec)
        if case["layout"] == "il":
            tl.tm_dslash_il(st["op"], st["out"], st["in"], n, **args)
        elif case["op"] == "hpe4":
            tl.tm_hpe_apply(st["op"], st["out"], st["in"], n, 4, prec)
        elif case["op"] == "g5DW":
            tl.tm_dslash_g5(st["op"], st["out"], st["in"], n, **args)
        else:
            tl.tm_dslash(st["op"], st["out"], st["in"], n, **args)
        return st["out"].view(_VIEW[case["prec"]])
    if kind == "solve":
        if case["layout"] == "il":
            tl.tm_cg_solve_il(st["op"], st["x"], st["eta"], n, st["params"])
        else:
            tl.tm_cg_solve(st["op"], st["x"], st["eta"], n, st["params"])
        return st["x"].view(torch.float64 if case["mode"] == "mixed" else _VIEW[case["prec"]])
    if kind == "momenta":
        tl.loop_contract_local_mom(L, st["left"], st["right"], prec, n, tl.LOOP_VV, st["mom"], st["out"])
        return st["out"]
    x, dw = st["x"], st["dw"]
    if case["layout"] == "il":
        tl.tm_dslash_il(st["op"], dw, x, n, mu_zero=True, prec=prec)
        for i, (mode, r, g5) in enumerate([(tl.LOOP_VV, x, False), (tl.LOOP_GEN, dw, True)]):
            tl.loop_contract_local_il(L, x, r, prec, n, mode, st["local"][i], right_g5=g5)
            tl.loop_contract_oneD_il(st["op"], x, r, prec, n, mode, st["oned"][i], right_g5=g5)
    else:
        if "x64" in st:
            tl.tm_spinor_convert(L, x, prec, st["x64"], tl.F64, n)
        tl.tm_dslash_g5(st["op"], dw, x, n, mu_zero=True, prec=prec)
        for i, (mode, r) in enumerate([(tl.LOOP_VV, x), (tl.LOOP_GEN, dw)]):
            tl.loop_contract_local(L, x, r, prec, n, mode, st["local"][i])
            tl.loop_contract_oneD(st["op"], x, r, prec, n, mode, st["oned"][i])
    return {"local": st["local"], "oneD": st["oned"]}


# ------------------------------------------------------------------ work
_SIZE = {"f64": 8, "ff": 8, "f32": 4, "f16": 2, "bf16": 2}


def _solve_work(V, n, e, schur, iters, mixed):
    """CG on the normal equations: per iteration two operator applications
    (each at least one vector in, one out) and r, x and p read and written
    once, the links twice; mixed solves also write x and read the source in
    FP64.  Schur solves keep half-lattice vectors."""
    field = 24.0 * V * n
    half = 0.5 if schur else 1.0
    links = 4 * 12.0 * V * e
    b = iters * (10 * half * field * e + 2 * links) + 2 * field * (8 if mixed else e)
    return b, iters * n * V * (2 * 1368.0 + half * 144.0)


def work(case):
    e, kind = _SIZE[case["prec"]], case["kind"]
    if kind == "group":
        w = [_solve_work(L[0] * L[1] * L[2] * L[3], n, e, True, case["iters"], False) for L, n, _, _ in _sets(case)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    L = _dims(case)
    V = L[0] * L[1] * L[2] * L[3]
    links = 4 * (12 if case["prec"] == "f32" else 18) * e * V
    if kind == "dslash":
        k = 4 if case["op"] == "hpe4" else 1
        return {"bytes": k * (2 * 24.0 * e * V * case["n"] + links), "flops": k * 1368.0 * V * case["n"]}
    if kind == "solve":
        b, f = _solve_work(V, case["n"], e, case["schur"], case["iters"], case["mode"] == "mixed")
        return {"bytes": b, "flops": f}
    if kind == "loops":  # D_W once; each contraction its two fields, the one-derivative ones the links
        n, field = case["n"], 24.0 * e * V * case["n"]
        out = 8.0 * 2 * n * L[3] * 2 * (16 + 64)
        return {"bytes": 2 * field + links + (2 + 4) * field + 2 * links + out + (2 * field if case["prec"] == "ff" else 0),
                "flops": n * V * (1368.0 + 2 * 384.0 + 2 * 4224.0)}
    if kind == "momenta":  # the 16 products once per site, then one phase multiply-add per momentum
        m = len(_momenta(case))
        return {"bytes": 2 * 24.0 * e * V * case["n"] + 16.0 * 16 * L[3] * m * case["n"],
                "flops": case["n"] * V * (384.0 + 16 * 8.0 * m)}
    lp = _solve_work(V, case["n_lp"] + case["n_hp"], e, True, 6, False)
    hp = _solve_work(V, case["n_hp"], 4, True, 32, True)
    loops = 8 * 24.0 * V * ((case["n_lp"] + case["n_hp"]) * e + case["n_hp"] * 8)  # D_W and the contractions' fields
    return {"bytes": lp[0] + hp[0] + loops,
            "flops": lp[1] + hp[1] + (case["n_lp"] + 2 * case["n_hp"]) * V * (1368.0 + 2 * 384.0 + 4224.0)}


# ------------------------------------------------------------------ tolerances
def tolerance(case):
    """About four times the distance from complex128 that was measured on a GB300 (in brackets)."""
    kind, prec = case["kind"], case["prec"]
    if kind == "dslash":
        # 16 bits: links and projections rounded to the format (2.6e-4, 2e-3);
        # FP32 (6e-8), FP64 (1.4e-16; the fourth-order expansion 6e-16);
        # float-float by its words, single high parts of which may round the
        # other way (5e-14)
        rel = {"f16": 1.2e-3, "bf16": 9e-3, "f32": 3e-7, "ff": 1e-9, "f64": 3e-15}[prec]
        return {"rel": rel, "max": 3e-7 if prec == "ff" else 30 * rel}
    if kind in ("solve", "group") and case.get("mode", "plain") == "mixed":
        return {"rel": 40 * case["tol"]}  # one iteration more or less
    if kind in ("solve", "group"):
        # truncated solves: the rounding of the 16-bit vectors (6.6e-4,
        # 5.3e-3), and now and then one iteration more or less of a system
        return {"rel": {"f16": 1e-2, "bf16": 2.2e-2, "f32": 4e-5, "f64": 1e-9}[prec]}
    if kind == "loops":  # (FP16 2.6e-4, float-float 1.8e-14)
        return {"rel": {"f16": 1.2e-3, "bf16": 1e-2, "f32": 1e-6, "ff": 2e-13, "f64": 1e-13}[prec]}
    if kind == "momenta":  # (FP32 2.1e-7)
        return {"rel": {"f16": 1e-6, "f32": 1e-6, "ff": 1e-11, "f64": 1e-12}[prec]}
    # estimates and errors from truncated solutions of a few sources (up to 1e-2)
    return {"rel": 3e-2}


# ------------------------------------------------------------------ complex128
# gamma_1 .. gamma_4 of the DeGrand-Rossi basis: row -> (column, phase)
_GAMMA = [[(3, 1j), (2, 1j), (1, -1j), (0, -1j)], [(3, -1), (2, 1), (1, 1), (0, -1)],
          [(2, 1j), (3, -1j), (0, -1j), (1, 1j)], [(2, 1), (3, 1), (0, 1), (1, 1)]]


def _gamma_matrices():
    g = torch.zeros((4, 4, 4), dtype=C128)
    for m, rows in enumerate(_GAMMA):
        for a, (b, ph) in enumerate(rows):
            g[m, a, b] = ph
    return g


def _shift(f, mu, step, axis0, anti=True):
    """f(x + step mu); axis0 the axis of t; antiperiodic in time where asked."""
    ax = axis0 + 3 - mu
    g = torch.roll(f, -step, dims=ax)
    if anti and mu == 3:
        g = g.clone()
        g.select(ax, g.shape[ax] - 1 if step > 0 else 0).neg_()
    return g


def _colour(U, chi, dag=False):
    """U chi (or U^dag chi) per site: U (T, Z, Y, X, 3, 3), chi (n, T, Z, Y, X, 4, 3)."""
    out = None
    for b in range(3):
        col = (U[..., b, :].conj() if dag else U[..., :, b]).unsqueeze(-2)
        term = col * chi[..., b:b + 1]
        out = term if out is None else out.add_(term)
    return out


def _one_minus_gamma(mu, sign, chi):
    """(1 + sign gamma_mu) chi."""
    out = chi.clone()
    for a, (b, ph) in enumerate(_GAMMA[mu]):
        out[..., a, :].add_(chi[..., b, :] * (sign * ph))
    return out


def _hops(U, psi, dag=False):
    s = 1 if dag else -1
    out = torch.zeros_like(psi)
    for mu in range(4):
        out += _one_minus_gamma(mu, s, _colour(U[mu], _shift(psi, mu, +1, 1)))
        out += _one_minus_gamma(mu, -s, _shift(_colour(U[mu], psi, dag=True), mu, -1, 1))
    return out


def _twist(psi, nu, inverse=False):
    """A psi = (1 + i nu gamma_5) psi, or A^-1 psi."""
    s = torch.tensor([1, 1, -1, -1], dtype=torch.float64, device=psi.device)[:, None] * (1j * nu)
    return psi * (1 - s) / (1 + nu * nu) if inverse else psi * (1 + s)


def _apply(U, psi, kappa, nu, dag=False):
    return _twist(psi, -nu if dag else nu) - kappa * _hops(U, psi, dag)


def _parity(L):
    X, Y, Z, T = L
    r = [torch.arange(e, device="cuda") for e in (T, Z, Y, X)]
    return (r[0][:, None, None, None] + r[1][:, None, None] + r[2][:, None] + r[3]) % 2


def _cg(U, eta, kappa, mu, tol, schur):
    """Per-system CG on the normal equations of M, or of the odd-site Schur complement."""
    nu = 2 * kappa * mu
    L = tuple(reversed(eta.shape[1:5]))
    odd = _parity(L).to(torch.float64)[None, ..., None, None]

    def op(v, dag=False):
        if not schur:
            return _apply(U, v, kappa, nu, dag)
        s = -nu if dag else nu
        w = _twist(_hops(U, v, dag) * (1 - odd), s, inverse=True)
        return _twist(v, s) - kappa * kappa * _hops(U, w, dag) * odd

    def norm2(v):
        return torch.view_as_real(v).square().sum(dim=tuple(range(1, v.dim() + 1)))

    def per(a, v):
        return a.view((-1,) + (1,) * (v.dim() - 1)) * v

    src = eta
    if schur:
        src = (eta + kappa * _hops(U, _twist(eta * (1 - odd), nu, inverse=True))) * odd
    r = op(src, True)
    del src
    b2 = rr = norm2(r)
    x, p = torch.zeros_like(r), r.clone()
    on = rr > tol * tol * b2
    for _ in range(2000):
        if not bool(on.any()):
            break
        t = op(p)
        al = torch.where(on, rr / norm2(t), torch.zeros_like(rr))
        x += per(al, p)
        r -= per(al, op(t, True))
        new = norm2(r)
        be = torch.where(on, new / rr, torch.ones_like(rr))
        rr = torch.where(on, new, rr)
        on = on & (rr > tol * tol * b2)
        p = torch.where(on.view((-1,) + (1,) * (p.dim() - 1)), r + per(be, p), p)
    if schur:
        x = x + _twist((eta + kappa * _hops(U, x)) * (1 - odd), nu, inverse=True)
    return x


def _philox_z4(L, seed, n):
    """Z4 sources 0 .. n - 1 of a seed: Philox4x32-10 keyed by the seed on (lexicographic site, source, 0, 0)."""
    X, Y, Z, T = L
    V, M32 = X * Y * Z * T, 0xFFFFFFFF
    c = [torch.arange(V, device="cuda").repeat(n), torch.arange(n, device="cuda").repeat_interleave(V)]
    c += [torch.zeros_like(c[0]), torch.zeros_like(c[0])]
    k = [seed & M32, (seed >> 32) & M32]

    def mul(m, v):  # high and low words of a 32 x 32-bit product
        lo, hi = (m & 0xFFFF) * v, (m >> 16) * v
        s = lo + ((hi & 0xFFFF) << 16)
        return (hi >> 16) + (s >> 32), s & M32

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & M32, (k[1] + 0xBB67AE85) & M32]
    ph = torch.tensor([1, 1j, -1, -1j], dtype=C128, device="cuda")
    q = (c[0][:, None] >> (2 * torch.arange(12, device="cuda"))) & 3
    return ph[q].view(n, T, Z, Y, X, 4, 3)


def _round(psi, prec):
    """The values as stored in the precision (two 32-bit words hold an FP64 value to 2^-48)."""
    if prec in ("f64", "ff"):
        return psi
    return torch.view_as_complex(torch.view_as_real(psi).to(_VIEW[prec]).to(torch.float64))


def _laid_out(psi, prec, layout):
    """Canonical spinors in the order of the library's fields, as FP64 numbers."""
    n, T, Z, Y, X = psi.shape[:5]
    V = T * Z * Y * X
    order = torch.argsort(_parity((X, Y, Z, T)).reshape(-1), stable=True)  # even sites, then odd ones
    f = psi.reshape(n, V, 12)[:, order].view(n, 2, V // 2, 12)
    if layout == "il":
        nb = (n + 15) // 16
        pad = torch.zeros((nb * 16, 2, V // 2, 12), dtype=C128, device=psi.device)
        pad[:n] = f
        pad = pad.view(nb, 16, 2, V // 2, 12)
        slots = torch.empty((12, 16), dtype=torch.long, device=psi.device)  # system of each slot of a row
        for k in range(12):
            for s in range(16):
                j = (s >> 1) ^ (4 if k % 3 == 2 else 0)
                slots[k, s] = j + 8 * (s & 1)
        out = torch.stack([pad[:, slots[k], :, :, k].permute(0, 2, 3, 1) for k in range(12)], dim=3)
        return torch.view_as_real(out.contiguous()).reshape(-1)
    r = torch.view_as_real(f)  # (n, 2, Vh, 12, 2)
    if prec == "ff":
        hi = r.to(torch.float32)
        r = torch.stack([hi.to(torch.float64), (r - hi).to(torch.float32).to(torch.float64)], dim=-1)
    per = 16 // _VIEW[prec].itemsize
    r = r.reshape(n, 2, V // 2, -1, per)
    return r.transpose(2, 3).reshape(-1)


def _dirac16(mode_g5):
    g = _gamma_matrices()
    out = torch.zeros((16, 4, 4), dtype=C128)
    for i in range(16):
        m = torch.eye(4, dtype=C128)
        for k in range(4):
            if (i >> k) & 1:
                m = m @ g[k]
        out[i] = m
    if mode_g5:
        out[:, 2:, :] *= -1
    return out.cuda()


def _bilinear(L, R):
    """sum over a slice and colour of conj(L_a) R_b: (n, T, 4, 4)."""
    n, T = L.shape[:2]
    l, r = (f.reshape(n * T, -1, 4, 3).transpose(1, 2).reshape(n * T, 4, -1) for f in (L, R))
    return torch.stack([torch.stack([(l[:, a].conj() * r[:, b]).sum(-1) for b in range(4)], -1)
                        for a in range(4)], -2).view(n, T, 4, 4)


def _project(S):
    """(n, ..., T, 4, 4) -> loops (n, ..., 16, T, 2) with P = gamma_5."""
    out = torch.einsum("gab,n...tab->n...gt", _dirac16(True), S)
    return torch.view_as_real(out.contiguous())


def _loops(U, L, R):
    """Local and one-derivative loops with P = gamma_5."""
    oned = []
    for mu in range(4):
        fwd = _bilinear(L, _colour(U[mu], _shift(R, mu, +1, 1)))
        bwd = _bilinear(L, _shift(_colour(U[mu], R, dag=True), mu, -1, 1))
        f2 = _bilinear(_shift(L, mu, +1, 1), _colour(U[mu], R, dag=True))
        Ub = _shift(U[mu], mu, -1, 0, anti=False)
        b2 = _bilinear(_shift(L, mu, -1, 1), _colour(Ub, R))
        oned.append(0.25 * (fwd - bwd - f2 + b2))
    return _project(_bilinear(L, R)), _project(torch.stack(oned, 1))


def _both_estimators(U, x, kappa):
    """[local vv, local gen], [oneD vv, oneD gen] of solutions x."""
    dw = _apply(U, x, kappa, 0.0)
    dw[..., 2:, :] *= -1  # gamma_5
    pairs = [_loops(U, x, x), _loops(U, x, dw)]
    return [p[0] for p in pairs], [p[1] for p in pairs]


def _combine(hp, lphp, lp, scale):
    hp, lphp, lp = (torch.view_as_complex(a.reshape(a.shape[0], -1, 2).contiguous()) * scale for a in (hp, lphp, lp))
    d = hp - lphp
    mean = d.mean(0) + lp.mean(0)
    if d.shape[0] < 2 or lp.shape[0] < 2:
        err = torch.full_like(mean, complex(float("nan"), float("nan")))
    else:
        v = [torch.view_as_real(a).var(0, unbiased=True) / a.shape[0] for a in (d, lp)]
        err = torch.view_as_complex((v[0] + v[1]).sqrt())
    return [torch.view_as_real(mean).reshape(-1).contiguous(), torch.view_as_real(err).reshape(-1).contiguous()]


def exact(case, seed):
    kind, prec = case["kind"], case["prec"]
    if kind == "group":
        out = []
        for i, (L, n, kappa, mu) in enumerate(_sets(case)):
            x = _cg(_gauge(L, seed + 100 * i), _philox_z4(L, seed + i, n), kappa, mu, case["tol"], True)
            out.append(_laid_out(x, prec, "std"))
        return out
    L = _dims(case)
    if kind == "momenta":
        l, r = (_round(_spinors(L, case["n"], seed, w), prec) for w in (2, 3))
        X, Y, Z, T = L
        out = []
        for q in _momenta(case):
            ang = (q[2] * torch.arange(Z, device="cuda")[:, None, None] / Z
                   + q[1] * torch.arange(Y, device="cuda")[:, None] / Y + q[0] * torch.arange(X, device="cuda") / X)
            ph = torch.exp(-2j * math.pi * ang.to(C128))
            out.append(_project(_bilinear(l, r * ph[None, None, ..., None, None])))
        return torch.stack(out, 1)
    U, kappa, mu = _gauge(L, seed), case.get("kappa", 0.161), case.get("mu", 0.003)
    nu = 2 * kappa * mu
    if kind == "dslash":
        psi = _round(_spinors(L, case["n"], seed), prec)
        if case["op"] == "hpe4":
            for _ in range(4):
                psi = _twist(-kappa * _hops(U, psi), nu, inverse=True)
        else:
            psi = _apply(U, psi, kappa, 0.0 if "DW" in case["op"] else nu, dag=case["op"] == "Mdag")
            if case["op"] == "g5DW":
                psi[..., 2:, :] *= -1
        return _laid_out(psi, prec, case["layout"])
    if kind == "solve":
        if case["n"] * L[0] * L[1] * L[2] * L[3] * case["iters"] > 7e8:
            return None  # minutes in complex128
        x = _cg(U, _philox_z4(L, seed, case["n"]), kappa, mu, case["tol"], case["schur"])
        return _laid_out(x, "f64" if case["mode"] == "mixed" else prec, case["layout"])
    if kind == "loops":
        x = _round(_spinors(L, case["n"], seed), prec)
        local, oned = _both_estimators(U, x, kappa)
        return {"local": local, "oneD": oned}
    n_hp, n_all = case["n_hp"], case["n_hp"] + case["n_lp"]
    res = {}
    for which, n, tol in (("lp", n_all, 1e-2), ("hp", n_hp, 1e-9)):
        parts = []
        eta = _philox_z4(L, seed, n)
        for b in range(0, n, 16):
            parts.append(_both_estimators(U, _cg(U, eta[b:b + 16], kappa, mu, tol, True), kappa))
        for i, op in enumerate(("local", "oneD")):
            for j, est in enumerate(("vv", "gen")):
                if "%s_%s" % (op, est) in TSM_KINDS:
                    res["%s_%s_%s" % (which, op, est)] = torch.cat([p[i][j] for p in parts]).reshape(n, -1)
    for k in TSM_KINDS:
        hp, lp = res["hp_" + k], res["lp_" + k]
        res["est_" + k] = _combine(hp, lp[:n_hp], lp[n_hp:], -2j * nu if k.endswith("vv") else 2.0)
    return res
