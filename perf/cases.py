"""Performance cases of the per-sample PEPS contraction (arXiv:1908.09359).

Each case is one pass through a public entry point of ``paper_1908_09359_gb300.api`` at a
size that occurs in use: the column steps and the fit's QR on their own (the blocks that
every sample is made of), and whole sweeps, measurements and sample steps.  Sizes come
from the workloads of ``paper_1908_09359_gb300.inputs`` (4x4 D2 Dc4, 8x8 D4 Dc16,
16x16 D6 Dc24, 24x24 D8 Dc32) and, for drawn cases, from the ranges they span.

``kind`` of a case:
  env3          three-line column step of n_chains chains (App. C), device tensors
  env3_noalloc  the same without a context (callers that must not allocate)
  env4          four-line column step of a row pair (App. C)
  qr            batched thin QR of the truncation fit (App. B)
  measure       fresh environments, E_loc, ln|Psi|, sign and one chain's d ln Psi
  sweep         one sequential Metropolis sweep of every chain (Eq. (9))
  step          one sample step: sweep, measurement, gradient; with ``update`` the
                sign-SGD step as well
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1908_09359_gb300 import api, inputs

LATTICE = 4  # lattice of the contexts that only run single column steps


def listed():
    return [
        # smallest call of the library: one FP32 column step for 64 chains of the 8x8
        # workload, by a caller that holds no context (a service with a planned pool)
        dict(name="noalloc_8x8", kind="env3_noalloc", precision="fp32", n=64, cT=16, cB=16, cT2=16, cB2=16,
             Dl=4, Dr=4, Du=4, Dd=4),
        # the step that sampling and the fit consist of, at the headline lattice's bulk
        # shape and chain count, in the precision production runs use (split BF16)
        dict(name="env3_split_24x24", kind="env3", precision="bf16x3", n=512, cT=32, cB=32, cT2=32, cB2=32,
             Dl=8, Dr=8, Du=8, Dd=8),
        # the same step in the default precision (FP32) at the 16x16 workload's shape
        dict(name="env3_fp32_16x16", kind="env3", precision="fp32", n=2048, cT=24, cB=24, cT2=24, cB2=24,
             Dl=6, Dr=6, Du=6, Dd=6),
        # a column near the lattice edge: unequal bonds, a ragged chain count, plain BF16
        dict(name="env3_bf16_ragged", kind="env3", precision="bf16", n=777, cT=32, cB=27, cT2=20, cB2=31,
             Dl=8, Dr=7, Du=8, Dd=5),
        # the dominant step of the measurement (vertical and diagonal terms of E_loc)
        dict(name="env4_split_24x24", kind="env4", precision="bf16x3", n=512, cT=32, cB=32, cT2=32, cB2=32,
             D1l=8, D1r=8, Du1=8, Dd1=8, D2l=8, D2r=8, Dd2=8, bmajor=True),
        # the four-line step of the 8x8 workload in FP32, environments in the plain order
        dict(name="env4_fp32_8x8", kind="env4", precision="fp32", n=1024, cT=16, cB=16, cT2=16, cB2=16,
             D1l=4, D1r=4, Du1=4, Dd1=4, D2l=4, D2r=4, Dd2=4, bmajor=False),
        # the fit's orthogonalisation: one bulk site of 512 chains at the headline shape
        dict(name="qr_24x24", kind="qr", n=512, rows=256, cols=32, col_major=False),
        # the right-to-left half-sweeps' QR (column-major) at the 16x16 shape, rows that
        # fill no power of two
        dict(name="qr_16x16_cols", kind="qr", n=2048, rows=144, cols=24, col_major=True),
        # one chain of the smallest lattice: a measurement that is all launches and latency
        dict(name="measure_4x4", kind="measure", precision="fp32", L=4, D=2, chi=4, n=1, J2=0.0, decay=0.0),
        # thermalisation: a sweep without measurement at the 16x16 shape in split BF16
        dict(name="sweep_16x16", kind="sweep", precision="bf16x3", L=16, D=6, chi=24, n=256, J2=0.0, decay=1.0),
        # a whole optimisation step of the 8x8 workload in the default precision, all chains
        dict(name="step_8x8", kind="step", precision="fp32", L=8, D=4, chi=16, n=1024, J2=0.0, decay=1.0,
             update=True),
        # the headline sample step (24x24 J1-J2 D8 Dc32, split BF16) with a quarter of the
        # headline's 512 chains, the share of one of four ranks
        dict(name="step_24x24", kind="step", precision="bf16x3", L=24, D=8, chi=32, n=128, J2=0.5, decay=1.0,
             update=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: column steps of any precision with bonds 1..D and 1..Dc, QRs of
    D Dc x Dc shapes up to Dc = 56, and whole calls on lattices of 4 to 12 sites a side."""
    kind = rng.choice(["env3", "env3", "env4", "env4", "qr", "qr", "env3_noalloc", "measure", "sweep", "step"])
    if kind in ("env3", "env3_noalloc", "env4"):
        prec = "fp32" if kind == "env3_noalloc" else rng.choice(["bf16x3", "bf16x3", "fp32", "bf16", "tf32"])
        D = rng.randint(2, 4 if kind == "env3_noalloc" else 8)
        chi = rng.randint(2 * D, 4 * D)
        n = _log_int(rng, 1, 64) if kind == "env3_noalloc" else _log_int(rng, 16, 2048 if kind == "env3" else 512)
        # most columns are bulk ones; the others have any bonds up to the maxima
        bulk = rng.random() < 0.5
        c = lambda: chi if bulk else rng.randint(1, chi)  # noqa: E731
        d = lambda: D if bulk else rng.randint(1, D)      # noqa: E731
        case = dict(kind=kind, precision=prec, n=n, cT=c(), cB=c(), cT2=c(), cB2=c())
        if kind == "env4":
            case.update(D1l=d(), D1r=d(), Du1=d(), Dd1=d(), D2l=d(), D2r=d(), Dd2=d(),
                        bmajor=prec in ("bf16", "bf16x3") and rng.random() < 0.7)
        else:
            case.update(Dl=d(), Dr=d(), Du=d(), Dd=d())
        return case
    if kind == "qr":
        cols = rng.randint(4, 32) if rng.random() < 0.8 else rng.randint(33, 56)
        rows = cols * rng.randint(1, 8) if cols <= 32 else cols * rng.randint(1, 5)
        return dict(kind="qr", n=_log_int(rng, 64, 2048), rows=rows, cols=cols, col_major=rng.random() < 0.5)
    prec = rng.choice(["fp32", "fp32", "bf16x3"])
    D = rng.randint(2, 5)
    case = dict(kind=kind, precision=prec, L=2 * rng.randint(2, 6), D=D, chi=rng.randint(2 * D, 4 * D),
                n=_log_int(rng, 1, 256), J2=rng.choice([0.0, 0.5]), decay=1.0)
    if kind == "step":
        case["update"] = rng.random() < 0.5
    return case


# --------------------------------------------------------------------------- inputs

def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _spins(g, n):
    return torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8)


def _decayed(x, *axes):
    """x with index i of each given axis scaled by exp(-i/8): bond spectra that decay, as
    in environments and MPS sites of a truncated contraction."""
    for a in axes:
        w = torch.exp(-torch.arange(x.shape[a], device=x.device, dtype=x.dtype) / 8)
        x = x * w.reshape([-1 if i == a else 1 for i in range(x.dim())])
    return x


def _arrays(case, seed):
    """Inputs of the single-step and QR cases, all float32 on the device."""
    g = torch.Generator(device="cuda").manual_seed(1908093590 + int(seed))
    n = case["n"]
    if case["kind"] == "qr":
        Y = _decayed(_randn(g, n, case["rows"], case["cols"]), 2)
        return dict(Y=(Y.transpose(1, 2) if case["col_major"] else Y).contiguous())
    cT, cB, cT2, cB2 = (case[k] for k in ("cT", "cB", "cT2", "cB2"))
    if case["kind"] == "env4":
        l1, r1, u1, d1, l2, r2, d2 = (case[k] for k in ("D1l", "D1r", "Du1", "Dd1", "D2l", "D2r", "Dd2"))
        E = _decayed(_randn(g, n, cT, l1, l2, cB), 1, 4)
        return dict(E=(E.permute(0, 4, 1, 2, 3) if case["bmajor"] else E).contiguous(),
                    T=_decayed(_randn(g, n, cT, u1, cT2), 1), A1=_decayed(_randn(g, 2, l1, u1, r1, d1), 1, 2),
                    s1=_spins(g, n), A2=_decayed(_randn(g, 2, l2, d1, r2, d2), 1, 2), s2=_spins(g, n),
                    B=_decayed(_randn(g, n, cB, d2, cB2), 1))
    l, r, u, d = (case[k] for k in ("Dl", "Dr", "Du", "Dd"))
    return dict(E=_decayed(_randn(g, n, cT, l, cB), 1, 3), T=_decayed(_randn(g, n, cT, u, cT2), 1),
                A=_decayed(_randn(g, 2, l, u, r, d), 1, 2), spins=_spins(g, n),
                B=_decayed(_randn(g, n, cB, d, cB2), 1))


def _lattice_inputs(case, seed):
    L, D, chi = case["L"], case["D"], case["chi"]
    s = 1908093590 + 1000 * int(seed)
    return (inputs.peps_tensors(L, L, D, s, normalise=True, bond_decay=case["decay"]),
            inputs.sketch(L, chi, D, s), inputs.start_spins(case["n"], L, L, s))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("measure", "sweep", "step"):
        L, D, chi = case["L"], case["D"], case["chi"]
        t, sk, sp = _lattice_inputs(case, seed)
        ctx = api.PepsVMC(L, L, D, chi, case["n"], t, sk, J1=1.0, J2=case["J2"], seed=int(seed) + 1,
                          precision=api.PRECISIONS[case["precision"]])
        # the autotuner picks by timing among kernels that round differently; runs that
        # have to be reproducible switch it off (FP32 kernels all round alike)
        if case["precision"] != "fp32":
            ctx.set_autotune(False)
        ctx.set_spins(sp)
        return dict(case=case, ctx=ctx, spins=sp, steps=0)
    x = _arrays(case, seed)
    st = dict(case=case, x=x)
    if kind == "qr":
        st["Q"] = torch.empty_like(x["Y"])
        return st
    n, cT2, cB2 = case["n"], case["cT2"], case["cB2"]
    if kind == "env4":
        shape = (n, cT2, case["D1r"], case["D2r"], cB2)
        if case["bmajor"]:
            shape = (n, cB2, cT2, case["D1r"], case["D2r"])
        st["dims"] = (n, case["cT"], case["cB"], cT2, cB2) + tuple(
            case[k] for k in ("D1l", "D1r", "Du1", "Dd1", "D2l", "D2r", "Dd2"))
    else:
        shape = (n, cT2, case["Dr"], cB2)
        st["dims"] = (n, case["cT"], case["cB"], cT2, cB2) + tuple(case[k] for k in ("Dl", "Dr", "Du", "Dd"))
    st["out"] = torch.empty(shape, dtype=torch.float32, device="cuda")
    if kind != "env3_noalloc":
        D, chi = max(st["dims"][5:]), max(st["dims"][1:5])
        ctx = api.PepsVMC(LATTICE, LATTICE, D, chi, n, inputs.peps_tensors(LATTICE, LATTICE, D, 1),
                          inputs.sketch(LATTICE, chi, D, 1), seed=1, precision=api.PRECISIONS[case["precision"]])
        if case["precision"] != "fp32":
            ctx.set_autotune(False)
        st["ctx"] = ctx
    return st


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "qr":
        api.qr_pos(s["x"]["Y"], s["Q"], col_major=case["col_major"])
        return s["Q"]
    if kind == "env3_noalloc":
        x = s["x"]
        api.env3_left_noalloc(x["E"], x["T"], x["A"], x["spins"], x["B"], s["out"], s["dims"])
        return s["out"]
    if kind == "env3":
        x = s["x"]
        s["ctx"].env3_left(x["E"], x["T"], x["A"], x["spins"], x["B"], s["out"], s["dims"])
        return s["out"]
    if kind == "env4":
        x = s["x"]
        s["ctx"].env4_left(x["E"], x["T"], x["A1"], x["s1"], x["A2"], x["s2"], x["B"], s["out"], s["dims"],
                           bmajor=case["bmajor"])
        return s["out"]
    ctx = s["ctx"]
    if kind == "measure":
        e, lp, sg = ctx.measure()
        return dict(eloc=e, logpsi=lp, sign=sg, grad0=ctx.chain_grad(0))
    if kind == "sweep":
        rate = ctx.sample_sweep(1)
        return dict(rate=rate, spins=ctx.get_spins())
    r = ctx.energy_and_grad(1)
    out = dict(eloc=r["eloc"], logpsi=r["logpsi"], sign=r["sign"], grad=r["grad"], spins=ctx.get_spins())
    if case["update"]:
        s["steps"] += 1
        ctx.update(1e-4, s["steps"])
        out["tensors"] = ctx.get_tensors()
    return out


# ----------------------------------------------------------------------------- work

def _mac3(cT, cB, cT2, cB2, l, r, u, d):
    return l * cB * u * cT2 * cT, cB * cT2 * r * d * l * u, cT2 * r * cB2 * cB * d


def _mac4(cT, cB, cT2, cB2, l1, r1, u1, d1, l2, r2, d2):
    return (l1 * l2 * cB * u1 * cT2 * cT, l2 * cB * cT2 * r1 * d1 * l1 * u1, cB * cT2 * r1 * r2 * d2 * l2 * d1,
            cT2 * r1 * r2 * cB2 * cB * d2)


def _lattice_macs(case):
    """Multiply-adds of one chain's pass, with every product that does not depend on a
    site's spin, or that two steps of one site share, counted once."""
    L, D, chi, nfit = case["L"], case["D"], case["chi"], 3

    def leg(i):
        return 1 if i in (0, L) else D

    def bond(k, m):  # bond m of the boundary MPS after k rows
        j = min(m, L - m)
        return 1 if k == 0 or j == 0 else min(chi, D ** min(j, 8), D ** min(8, k * 1))

    def fit(k):  # row k absorbed and truncated
        t = 0
        for m in range(L):
            s = _mac3(bond(k, m), bond(k + 1, m), bond(k, m + 1), bond(k + 1, m + 1), leg(m), leg(m + 1), leg(k),
                      leg(k + 1))
            t += sum(s) + nfit * (sum(s) + s[2])
        return t

    def steps3(k, pair):
        t = 0
        for m in range(L):
            s = _mac3(bond(k, m), bond(L - 1 - k, m), bond(k, m + 1), bond(L - 1 - k, m + 1), leg(m), leg(m + 1),
                      leg(k), leg(k + 1))
            t += s[0] + (2 if pair else 1) * (s[1] + s[2])
        return t

    def steps4(k):
        t = 0
        for m in range(L):
            s = _mac4(bond(k, m), bond(L - 2 - k, m), bond(k, m + 1), bond(L - 2 - k, m + 1), leg(m), leg(m + 1),
                      leg(k), leg(k + 1), leg(m), leg(m + 1), leg(k + 2))
            t += sum(s)                                                    # right environments
            if case["J2"] != 0.0:
                t += s[0] + 2 * s[1] + 4 * (s[2] + s[3]) + 2 * sum(s)      # four variants, two diagonals
            else:
                t += s[0] + 2 * (s[1] + s[2] + s[3])
        return t

    fits = sum(fit(k) for k in range(L - 1))
    sweep = 2 * (2 * fits + sum(2 * steps3(k, True) for k in range(L)))
    measure = fits * (1 if case["kind"] == "step" else 2)
    measure += sum(2 * steps3(k, True) + steps3(k, False) for k in range(L)) + sum(steps4(k) for k in range(L - 1))
    return {"measure": measure, "sweep": sweep, "step": sweep + measure}[case["kind"]]


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "qr":
        m, c = case["rows"], case["cols"]
        return dict(bytes=8.0 * n * m * c, flops=2.0 * n * (2.0 * m * c * c - 2.0 * c ** 3 / 3.0))
    if kind in ("measure", "sweep", "step"):
        L, D = case["L"], case["D"]
        P = inputs.n_params(L, L, D)
        out = {"measure": 17.0 * n + 8.0 * P / 2, "sweep": float(n * L * L),
               "step": 17.0 * n + 8.0 * P + n * L * L + (8.0 * P if case.get("update") else 0.0)}[kind]
        return dict(bytes=8.0 * P + n * L * L + out, flops=2.0 * n * _lattice_macs(case))
    cT, cB, cT2, cB2 = (case[k] for k in ("cT", "cB", "cT2", "cB2"))
    if kind == "env4":
        l1, r1, u1, d1, l2, r2, d2 = (case[k] for k in ("D1l", "D1r", "Du1", "Dd1", "D2l", "D2r", "Dd2"))
        per = cT * l1 * l2 * cB + cT * u1 * cT2 + cB * d2 * cB2 + cT2 * r1 * r2 * cB2
        site = 2 * (l1 * u1 * r1 * d1 + l2 * d1 * r2 * d2)
        macs = sum(_mac4(cT, cB, cT2, cB2, l1, r1, u1, d1, l2, r2, d2))
    else:
        l, r, u, d = (case[k] for k in ("Dl", "Dr", "Du", "Dd"))
        per = cT * l * cB + cT * u * cT2 + cB * d * cB2 + cT2 * r * cB2
        site = 2 * l * u * r * d
        macs = sum(_mac3(cT, cB, cT2, cB2, l, r, u, d))
    return dict(bytes=4.0 * (n * per + site) + n, flops=2.0 * n * macs)


# ---------------------------------------------------------------------------- exact

def _exact_measure(case, seed):
    """E_loc, ln|Psi|, sign and chain 0's d ln Psi by full contraction (the truncation is
    exact once Dc >= D^(L/2)), row by row over the D^L boundary vector."""
    L, D = case["L"], case["D"]
    t, _, spins = _lattice_inputs(case, seed)
    A, off = [], 0
    for k in range(L):
        for m in range(L):
            shp = inputs.site_shape(L, L, D, k, m)
            size = int(np.prod(shp))
            A.append(torch.from_numpy(t[off:off + size].reshape(shp)))
            off += size

    def psi(sites):
        v = torch.ones([1] * (L + 1), dtype=torch.float64)  # upper legs, then the row's running bond
        for k in range(L):
            for m in range(L):
                a = sites[k * L + m]  # (l, r, u, d); the leading axis of v is the current upper leg
                v = torch.tensordot(v, a, dims=([0, L], [2, 0]))  # -> other legs, r, d
                v = v.movedim(-1, L - 1)                           # d joins the legs, r stays last
        return v.reshape(())

    def select(s):
        return [A[i][0 if s[i] > 0 else 1] for i in range(L * L)]

    e, lp, sg = [], [], []
    for c in range(case["n"]):
        s = spins[c].reshape(-1).astype(int)
        p0 = psi(select(s))
        pairs = [(k * L + m, k * L + m + 1, 1.0) for k in range(L) for m in range(L - 1)]
        pairs += [(k * L + m, (k + 1) * L + m, 1.0) for k in range(L - 1) for m in range(L)]
        if case["J2"] != 0.0:
            for k in range(L - 1):
                for m in range(L - 1):
                    pairs += [(k * L + m, (k + 1) * L + m + 1, case["J2"]), (k * L + m + 1, (k + 1) * L + m, case["J2"])]
        tot = 0.0
        for i, j, J in pairs:
            tot += J * 0.25 * s[i] * s[j]
            if s[i] != s[j]:
                q = s.copy()
                q[i], q[j] = s[j], s[i]
                tot += J * 0.5 * float(psi(select(q)) / p0)
        e.append(tot)
        lp.append(float(torch.log(torch.abs(p0))))
        sg.append(1 if float(p0) > 0 else -1)
    sites = [a.clone().requires_grad_(True) for a in select(spins[0].reshape(-1).astype(int))]
    p0 = psi(sites)
    grads = torch.autograd.grad(p0, sites)
    g0 = torch.cat([(g / p0.detach()).reshape(-1) for g in grads])
    return dict(eloc=np.array(e), logpsi=np.array(lp), sign=np.array(sg, dtype=np.int8), grad0=g0.numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("measure", "sweep", "step"):
        # a truncated contraction has no value apart from the method's own arithmetic
        if kind == "measure" and case["L"] == 4 and case["D"] == 2 and case["chi"] >= 4 and case["n"] <= 16:
            return _exact_measure(case, seed)
        return None
    x = {k: (v.double() if v.dtype == torch.float32 else v) for k, v in _arrays(case, seed).items()}
    if kind == "qr":
        Y = x["Y"].transpose(1, 2) if case["col_major"] else x["Y"]
        Q, R = torch.linalg.qr(Y)
        sign = torch.where(torch.diagonal(R, dim1=1, dim2=2) < 0, -1.0, 1.0).to(Q.dtype)
        Q = Q * sign[:, None, :]
        return (Q.transpose(1, 2) if case["col_major"] else Q).contiguous()
    slot = lambda s: (s < 0).long()  # noqa: E731
    out = []
    for i in range(0, case["n"], 64):
        c = slice(i, min(i + 64, case["n"]))
        if kind == "env4":
            E = x["E"][c].permute(0, 2, 3, 4, 1) if case["bmajor"] else x["E"][c]
            X = torch.einsum("nalmb,naux->nlmbux", E, x["T"][c])
            Y = torch.einsum("nlmbux,nlurd->nmbxrd", X, x["A1"][slot(x["s1"][c])])
            Z = torch.einsum("nmbxrd,nmdse->nbxrse", Y, x["A2"][slot(x["s2"][c])])
            o = torch.einsum("nbxrse,nbey->nxrsy", Z, x["B"][c])
            out.append(o.permute(0, 4, 1, 2, 3) if case["bmajor"] else o)
        else:
            X = torch.einsum("nalb,naux->nlbux", x["E"][c], x["T"][c])
            Y = torch.einsum("nlbux,nlurd->nbxrd", X, x["A"][slot(x["spins"][c])])
            out.append(torch.einsum("nbxrd,nbdy->nxry", Y, x["B"][c]))
    return torch.cat(out).contiguous()
