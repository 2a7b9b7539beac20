"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one of five kinds of call, each through the public entry points (`api.ACSE`, the ctypes binding
of the C ABI for what the wrapper has no method for):

  drive     ACSE.run_until_stop: the framework's own driver of a trajectory from a reference 2-RDM
            (fixed step or line search), which reads E and ||A||^2 back after every step;
  steps     a few Euler steps from the reference on a stream of the caller's, nothing read back (what
            a driver of the user's own does; the scalar outputs are buffers that it keeps);
  residual  one residual A and ||A||^2 into buffers that the caller keeps;
  batch     the 2-RDMs of several instances of uneven r loaded, advanced by graph replays and read back;
  adjoint   the gradient of wE E(D_n) + wN ||A(D_n)||^2 along n checkpointed steps.

Inputs: synthetic integrals as in `acse_inputs.make_integrals` (drawn on the GPU), a small exact CAS state
above a doubly occupied core (`acse_inputs.cas_rdm_blocks` on the active orbitals, embedded here) or the
Hartree-Fock determinant, and then a rotation of all orbitals by a small random angle, so that the 2-RDM
is dense, as it is along any trajectory, and still that of an exact state.

`exact` evaluates the same quantities with plain torch float64 matrix products: the factored form of the
contraction (Appendices B and C) block by block in the spin, the Nakatsuji-Yasuda term in spin orbitals,
gradients by torch.autograd.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import acse_inputs as I
from paper_2604_02550_gb300 import _lib, api

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest problem of the test systems: r = 8, N = 8, Hartree-Fock start, 20 fixed steps in
        # plain FP64 -- what a first run looks like; launches and read-backs count
        dict(name="drive_fp64_r8", kind="drive", prec="fp64", r=8, n=8, cas=0, cap=20, ls=False, eps=1e-3),
        # r = 24, N = 12, CAS(6e,6o), line search, plain FP64: the mid-size reference run
        dict(name="drive_ls_fp64_r24", kind="drive", prec="fp64", r=24, n=12, cas=6, cap=2, ls=True, eps=1e-3),
        # the headline workload, r = 48, N = 20, in split-precision BF16
        dict(name="steps_bf16x3_r48", kind="steps", prec="bf16x3", r=48, n=20, cas=6, nsteps=2, singlet=False,
             eps=1e-4, recon="V"),
        # the TF32 variant of that precision at an r that is no multiple of 16
        dict(name="steps_tf32x3_r40", kind="steps", prec="tf32x3", r=40, n=16, cas=6, nsteps=2, singlet=False,
             eps=1e-4, recon="V"),
        # the largest r that the library takes, with the closed-shell specialisation
        dict(name="steps_bf16x3_singlet_r64", kind="steps", prec="bf16x3", r=64, n=24, cas=6, nsteps=1, singlet=True,
             eps=1e-4, recon="V"),
        # an odd size: one residual in split precision, as a scan over geometries evaluates
        dict(name="residual_bf16x3_r31", kind="residual", prec="bf16x3", r=31, n=14, cas=6, recon="V"),
        # the FP64-accurate precision to a converged energy: line-searched steps at r = 48
        dict(name="drive_ls_ozaki_r48", kind="drive", prec="ozaki", r=48, n=20, cas=6, cap=2, ls=True, eps=1e-4),
        # the same precision on a ragged size
        dict(name="residual_ozaki_r30", kind="residual", prec="ozaki", r=30, n=12, cas=6, recon="V"),
        # the Nakatsuji-Yasuda reconstruction
        dict(name="steps_ny_bf16x3_r32", kind="steps", prec="bf16x3", r=32, n=14, cas=6, nsteps=1, singlet=False,
             eps=1e-4, recon="NY"),
        # 16 independent instances of uneven r, ground state and another of each size, advanced together
        dict(name="batch16_bf16x3", kind="batch", prec="bf16x3", rs="12,12,16,16,20,20,24,24,28,28,32,32,36,36,40,40",
             nsteps=8, eps=1e-4),
        # the adjoint of the r = 32 system over four checkpointed steps, FP64-accurate on the tensor cores
        dict(name="adjoint_ozaki_r32", kind="adjoint", prec="ozaki", r=32, n=14, cas=6, nsteps=4, eps=1e-4),
        # the adjoint in plain FP64, of a size that a check against finite differences uses
        dict(name="adjoint_fp64_r14", kind="adjoint", prec="fp64", r=14, n=8, cas=4, nsteps=2, eps=1e-3),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _system(rng, r):
    """Electron count and active space for r orbitals, within N <= r."""
    cas = 6 if r >= 16 and rng.random() < 0.7 else 4
    if r < 8 or rng.random() < 0.1:
        cas = 0
    lo = max(4, cas)
    return dict(n=2 * rng.randint(lo // 2, max(lo // 2, r // 4)), cas=cas)


def draw(rng):
    kind = rng.choice(["drive", "drive", "steps", "steps", "steps", "residual", "residual", "batch", "adjoint"])
    if kind == "drive":
        prec = rng.choice(["fp64", "ozaki"])
        r = _log_int(rng, 6, 22) if prec == "fp64" else _log_int(rng, 9, 46)
        ls = rng.random() < 0.5
        return dict(kind=kind, prec=prec, r=r, cap=rng.randint(1, 2) if r > 16 else rng.randint(2, 12), ls=ls,
                    eps=1e-4 if r >= 32 else 1e-3, **_system(rng, r))
    if kind == "steps":
        ny = rng.random() < 0.2
        prec = rng.choice(["bf16x3", "bf16x3", "tf32x3", "tf32"]) if not ny else rng.choice(["bf16x3", "tf32x3"])
        r = _log_int(rng, 9, 32 if ny else 62)
        return dict(kind=kind, prec=prec, r=r, nsteps=rng.randint(1, 3), singlet=rng.random() < 0.25,
                    eps=1e-4 if r >= 32 else 1e-3, recon="NY" if ny else "V", **_system(rng, r))
    if kind == "residual":
        prec = rng.choice(["bf16x3", "ozaki", "fp64", "tf32x3"])
        r = _log_int(rng, 9, {"fp64": 26, "ozaki": 56}.get(prec, 62))
        return dict(kind=kind, prec=prec, r=r, recon="V", **_system(rng, r))
    if kind == "batch":
        rs = [rng.choice([12, 15, 16, 20, 21, 24, 28, 32, 33, 36, 40]) for _ in range(rng.randint(3, 14))]
        return dict(kind=kind, prec=rng.choice(["bf16x3", "bf16x3", "tf32"]), rs=",".join(map(str, rs)),
                    nsteps=rng.randint(2, 6), eps=1e-4)
    prec = rng.choice(["ozaki", "ozaki", "fp64", "bf16x3"])
    r = _log_int(rng, 8, 14 if prec == "fp64" else 32)
    return dict(kind=kind, prec=prec, r=r, nsteps=rng.randint(1, 3), eps=1e-4 if r >= 32 else 1e-3, **_system(rng, r))


# --------------------------------------------------------------------------------------- inputs
def _integrals(r, gen):
    diag = torch.sort(torch.rand(r, generator=gen, device=DEV, dtype=F64) * 3.0 - 2.0).values
    off = torch.triu(torch.randn(r, r, generator=gen, device=DEV, dtype=F64) * 0.05, 1)
    h = off + off.T + torch.diag(diag)
    g = torch.randn(3 * r, r, r, generator=gen, device=DEV, dtype=F64) * 0.5
    scale = 0.5 ** torch.arange(3 * r, device=DEV, dtype=F64)
    b = (scale[:, None, None] * 0.5 * (g + g.transpose(1, 2))).reshape(3 * r, r * r)
    return h, (b.T @ b).reshape(r, r, r, r)


def _wedge(a, b):
    return 0.5 * (torch.einsum("ik,jl->ijkl", a, b) - torch.einsum("jk,il->ijkl", a, b))


def _rotate(x, u):
    for _ in range(4):   # each pass transforms the first index and moves it to the end
        r = u.shape[0]
        x = (x.reshape(r, -1).T @ u).reshape(r, r, r, r)
    return x.contiguous()


def _reference(r, n, cas, h, V, gen, root=0):
    """2-RDM blocks (aa, ab, bb): a CAS state (or, cas = 0, the determinant) above a core of the lowest
    orbitals, in orbitals rotated by a small random angle."""
    na = n // 2
    core = na - cas // 2
    t = torch.zeros(r, r, device=DEV, dtype=F64)
    t[range(core), range(core)] = 1.0
    if cas:
        act = slice(core, core + cas)
        hc = h[act, act].clone()
        for c in range(core):
            hc += 2.0 * V[act, act, c, c] - V[act, c, c, act]
        res = I.cas_rdm_blocks(hc.cpu().numpy(), V[act, act, act, act].cpu().numpy(), [], range(cas), cas, root=root)
        daa, dab, dbb = (torch.from_numpy(x).to(DEV) for x in (res.Daa, res.Dab, res.Dbb))
        ga, gb = ((2.0 / (cas - 1)) * (torch.einsum("pqrq->pr", s) + torch.einsum(e, dab))
                  for s, e in ((daa, "pqrq->pr"), (dbb, "qpqr->pr")))
        ta, tb = t.clone(), t.clone()
        ta[act, act], tb[act, act] = ga, gb
        aa, bb = _wedge(ta, ta), _wedge(tb, tb)
        ab = 0.5 * torch.einsum("ik,jl->ijkl", ta, tb)
        aa[act, act, act, act] += daa - _wedge(ga, ga)
        bb[act, act, act, act] += dbb - _wedge(gb, gb)
        ab[act, act, act, act] += dab - 0.5 * torch.einsum("ik,jl->ijkl", ga, gb)
    else:
        t[range(na), range(na)] = 1.0
        aa, ab = _wedge(t, t), 0.5 * torch.einsum("ik,jl->ijkl", t, t)
        bb = aa.clone()
    k = torch.randn(r, r, generator=gen, device=DEV, dtype=F64) * 0.02
    u = torch.matrix_exp(k - k.T)
    return tuple(_rotate(x, u) for x in (aa, ab, bb))


def _problem(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1_000_003 * (seed % 1_000_000) + case["r"])
    h, V = _integrals(case["r"], gen)
    return h, V, _reference(case["r"], case["n"], case["cas"], h, V, gen, case.get("root", 0))


def _instances(case):
    """The batch's instances: N = r/2 (even), CAS(4e,4o); every second one of a size takes the second root."""
    out = []
    for k, r in enumerate(int(x) for x in case["rs"].split(",")):
        out.append(dict(r=r, n=max(4, (r // 2) & ~1), cas=4, root=k % 2))
    return out


class _Inputs:
    """Integrals and electron counts as acse_batch_create takes them."""

    def __init__(self, r, n, h, V):
        self.r, self.n_alpha, self.n_beta, self.h, self.V = r, n // 2, n // 2, h, V


class _Batch:
    """A batch handle, freed with its owner."""

    def __init__(self, probs, prec):
        self.handle = _lib.acse_batch_create(probs, prec)

    def __del__(self):
        _lib.acse_batch_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs, D = [], []
        for i, inst in enumerate(_instances(case)):
            h, V, d = _problem(inst, seed + 7919 * i)
            probs.append(_Inputs(inst["r"], inst["n"], h, V))
            D.append(d)
        torch.cuda.synchronize()
        return dict(case=case, batch=_Batch(probs, case["prec"]), n=len(D), D=D,
                    out=[tuple(torch.empty_like(x) for x in d) for d in D])
    h, V, D0 = _problem(case, seed)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    kw = {}
    if kind == "drive":
        kw = dict(line_search=case["ls"], eps0=case["eps"])
    elif kind in ("steps", "residual"):
        kw = dict(recon=case["recon"], singlet=case.get("singlet", False))
    ctx = api.ACSE(case["r"], case["n"] // 2, case["n"] // 2, h, V, case["prec"], stream=stream, **kw)
    s = dict(case=case, ctx=ctx, stream=stream, D0=D0)
    if kind in ("drive", "steps"):
        s["D"] = tuple(x.clone() for x in D0)
    if kind == "steps":
        s["scalars"] = torch.empty(3, dtype=F64, device=DEV)
    if kind == "residual":
        s["A"] = ctx.zeros_blocks()
        s["norm2"] = torch.empty(1, dtype=F64, device=DEV)
    if kind == "adjoint":   # the checkpoints that the forward run leaves
        with torch.cuda.stream(stream):
            D = tuple(x.clone() for x in D0)
            s["ckpt"] = [D0]
            for _ in range(case["nsteps"]):
                ctx.step(D, case["eps"])
                s["ckpt"].append(tuple(x.clone() for x in D))
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------------------------ run
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        b = s["batch"].handle
        for i, d in enumerate(s["D"]):
            _lib.acse_batch_set_D(b, i, *d, case["eps"])
        E, n2, _, _ = _lib.acse_batch_run(b, s["n"], case["nsteps"], stop_rule=False)
        for i, d in enumerate(s["out"]):
            _lib.acse_batch_get_D(b, i, *d)
        return dict(E=E, norm2=n2, D=s["out"])
    ctx = s["ctx"]
    with torch.cuda.stream(s["stream"]):
        if kind == "drive":
            for dst, src in zip(s["D"], s["D0"]):
                dst.copy_(src)
            got = ctx.run_until_stop(s["D"], case["cap"], case["eps"])
            return dict(E=np.array(got["E"]), norm2=np.array(got["norm2"]), eps=np.array(got["eps"]),
                        E_stop=got["E_stop"], D=s["D"])
        if kind == "steps":
            for dst, src in zip(s["D"], s["D0"]):
                dst.copy_(src)
            sc = s["scalars"]
            for _ in range(case["nsteps"]):
                _lib.acse_step(ctx.ctx, *s["D"], case["eps"], sc[0:1], sc[1:2], sc[2:3])
            return dict(D=s["D"], E=sc[0:1], norm2=sc[1:2], eps=sc[2:3])
        if kind == "residual":
            _lib.acse_residual(ctx.ctx, *s["D0"], *s["A"], s["norm2"])
            return dict(A=s["A"], norm2=s["norm2"])
        dh, dV, dD = ctx.backward(s["ckpt"], case["nsteps"], case["eps"], wE=1.0, wN=0.01)
        return dict(dh=dh, dV=dV, dD=dD)


# ----------------------------------------------------------------------------------------- work
def _pass_flops(r, packed, singlet=False):
    """2 M N K of the O(r^6) products of one contraction pass, those of the same-spin pairs on i < j."""
    R, P = r * r, r * (r - 1) // 2
    if not packed:
        P = R
    if singlet:
        return 2 * ((2 * P) * P * P + (2 * R) * R * R + R * (2 * R) * (2 * R) + R ** 3)
    return 2 * (2 * (2 * P) * P * P + (2 * R) * R * R + (2 * R) ** 3 + 2 * R ** 3)


_MODULI = (127, 125, 123, 121, 119, 113, 109, 107, 103, 101, 97, 89, 83, 79, 73, 71, 67, 61, 59)


def _products(prec, r):
    """Tensor-core products of one real product in each precision."""
    if prec == "ozaki":
        need, p, t = (2 * r * r) << 98, 1, 0
        while p < need:
            p, t = p * _MODULI[t], t + 1
        return t
    return {"fp64": 1, "tf32": 1, "bf16x3": 3, "tf32x3": 3}[prec]


def work(case):
    kind, prec = case["kind"], case["prec"]
    if kind == "batch":
        sub = [dict(kind="steps", prec=prec, recon="V", singlet=False, nsteps=case["nsteps"], **i)
               for i in _instances(case)]
        w = [work(x) for x in sub]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    r = case["r"]
    blocks = 3 * 8 * r ** 4
    flops = _pass_flops(r, True, case.get("singlet", False)) * _products(prec, r)
    if case.get("recon") == "NY":
        flops += 120 * r ** 6 * _products(prec, r)
    if kind == "residual":           # D and K in, A out
        return {"bytes": 3 * blocks, "flops": flops}
    if kind == "steps":              # D and K in, D out, every step
        return {"bytes": 3 * blocks * case["nsteps"], "flops": 2 * flops * case["nsteps"]}
    if kind == "drive":
        return {"bytes": 3 * blocks * case["cap"], "flops": (4 if case["ls"] else 2) * flops * case["cap"]}
    # adjoint: per step the residual again, two W products and one D product of each of its two passes
    n = case["nsteps"]
    return {"bytes": blocks * (n + 1) + blocks + 2 * 8 * r ** 4, "flops": flops * (9 * n + 5)}


# ---------------------------------------------------------------------------------------- exact
# Spin-orbital pair tensors as dicts of r^4 blocks by the spins of their four indices.
def _spin_blocks(aa, ab, bb):
    return {"aaaa": aa, "bbbb": bb, "abab": ab, "baba": ab.permute(1, 0, 3, 2), "abba": -ab.permute(0, 1, 3, 2),
            "baab": -ab.permute(1, 0, 2, 3)}


def _con(eq, a, b):
    """A two-operand contraction of r^4 blocks as one matrix product."""
    ins, out = eq.split("->")
    x, y = ins.split(",")
    summed = [c for c in x if c in y]
    fx, fy = [c for c in x if c not in summed], [c for c in y if c not in summed]
    size = dict(zip(x, a.shape)) | dict(zip(y, b.shape))
    k = math.prod(size[c] for c in summed)
    A = a.permute([x.index(c) for c in fx + summed]).reshape(-1, k)
    B = b.permute([y.index(c) for c in summed + fy]).reshape(k, -1)
    C = (A @ B).reshape([size[c] for c in fx + fy])
    return C.permute([(fx + fy).index(c) for c in out])


def _exact_K(h, V, N):
    r = h.shape[0]
    eye = torch.eye(r, device=h.device, dtype=h.dtype)
    g = V.permute(0, 2, 1, 3)
    f = 1.0 / (2.0 * (N - 1))
    one = f * (torch.einsum("pr,qs->pqrs", h, eye) + torch.einsum("qs,pr->pqrs", h, eye))
    ab = 0.5 * g + one
    aa = 0.5 * (g - g.permute(0, 1, 3, 2)) + one - one.permute(0, 1, 3, 2)
    return aa, ab, aa


def _exact_gamma_M(D, N):
    f = 2.0 / (N - 1)
    g = {"a": f * (torch.einsum("pqrq->pr", D[0]) + torch.einsum("pqrq->pr", D[1])),
         "b": f * (torch.einsum("pqrq->pr", D[2]) + torch.einsum("qpqr->pr", D[1]))}
    gg = (_wedge(g["a"], g["a"]), 0.5 * torch.einsum("ik,jl->ijkl", g["a"], g["b"]), _wedge(g["b"], g["b"]))
    delta = tuple(d - w for d, w in zip(D, gg))
    return g, _spin_blocks(*(3.0 * d + w for d, w in zip(delta, gg))), delta


def _exact_B(W, M, g):
    """sum_{pqr} W^{kp}_{rq} 3D^{ijp}_{rql} with the Valdemoro 3D, by the spins of (i, j, k, l)."""
    X = {}   # X^{ij}_{kp} = sum_{rq} M^{ij}_{rq} W^{kp}_{rq}
    for t, f in (("aaaa", 1.0), ("bbbb", 1.0), ("abab", 2.0)):
        X[t] = f * _con("ijrq,kprq->ijkp", M[t], W[t])
    X["abba"] = -X["abab"].permute(0, 1, 3, 2)
    X["baba"] = X["abab"].permute(1, 0, 3, 2)
    X["baab"] = -X["abab"].permute(1, 0, 2, 3)
    w = {"a": torch.einsum("kprq,pr->kq", W["aaaa"], g["a"]) + torch.einsum("kprq,pr->kq", W["abba"], g["b"]),
         "b": torch.einsum("kprq,pr->kq", W["bbbb"], g["b"]) + torch.einsum("kprq,pr->kq", W["baab"], g["a"])}
    Q = {"a": torch.einsum("ipkp->ki", X["aaaa"]) + torch.einsum("ipkp->ki", X["abab"]),
         "b": torch.einsum("ipkp->ki", X["bbbb"]) + torch.einsum("ipkp->ki", X["baba"])}
    Z = {t: _con("kprq,jr->kpjq", W[t], g[t[2]]) for t in W}   # by the spins of (k, p, j, q)
    E = {}
    for t in W:                                     # spins of (i, j, k, l)
        i, j, k, l = t
        e = 0.0
        for p in "ab":
            for q in "ab":
                if k + p + j + q in Z and i + p + l + q in M:
                    e = e + 2.0 * _con("kpjq,iplq->kjil", Z[k + p + j + q], M[i + p + l + q]).permute(2, 1, 0, 3)
        if i == k:
            e = e - torch.einsum("ki,jl->ijkl", Q[k], g[l])
        E[t] = e
    B = {}
    for t in ("aaaa", "bbbb", "abab", "abba"):
        i, j, k, l = t
        t1 = _con("ijkp,pl->ijkl", X[t], g[l])
        t2 = 2.0 * _con("kq,ijlq->ijkl", w[k], M[i + j + l + k])
        B[t] = (t1 - t2 + E[t] - E[j + i + k + l].permute(1, 0, 2, 3)) / 9.0
    return B


def _to_spin_orbital(x):
    r = x["aaaa"].shape[0]
    out = torch.zeros((2 * r,) * 4, device=x["aaaa"].device, dtype=F64)
    for t, v in x.items():
        out[tuple(slice(0, r) if c == "a" else slice(r, 2 * r) for c in t)] = v
    return out


def _exact_ny(W, delta, r, n):
    """The same contraction with the Nakatsuji-Yasuda 3-cumulant, whose nine terms fall into four."""
    w, d = _to_spin_orbital(W), _to_spin_orbital(_spin_blocks(*delta))
    sig = -torch.ones(2 * r, device=DEV, dtype=F64)
    sig[:n // 2] = 1.0
    sig[r:r + n // 2] = 1.0
    x = _con("iarq,kprq->iakp", d, w)
    s3 = _con("ka,jial->ijkl", torch.einsum("pakp->ka", x) * sig, d)
    s1 = _con("iakp,jpal->ijkl", x * sig[None, :, None, None], d)
    del x
    y = _con("kprq,jpar->kqja", w, d) * sig
    s4 = _con("kqja,ialq->kjil", y, d).permute(2, 1, 0, 3)
    y = _con("kprq,palq->krla", w, d) * sig
    s6 = _con("krla,jiar->klji", y, d).permute(3, 2, 0, 1)
    del y
    e = s1 - 2.0 * s4
    T = (4.0 / 6.0) * (e - e.permute(1, 0, 2, 3) - s3 + 2.0 * s6)
    a, b = slice(0, r), slice(r, 2 * r)
    return {"aaaa": T[a, a, a, a], "bbbb": T[b, b, b, b], "abab": T[a, b, a, b], "abba": T[a, b, b, a]}


def _exact_G(Wb, D, case, s):
    """<[a+_i a+_j a_l a_k, W^]> for W with W^T = s W: blocks (aa, ab, bb)."""
    g, M, delta = _exact_gamma_M(D, case["n"])
    W = _spin_blocks(*Wb)
    B = _exact_B(W, M, g)
    if case.get("recon") == "NY":
        ny = _exact_ny(W, delta, case["r"], case["n"])
        B = {t: B[t] + ny[t] for t in B}
    out = []
    for t, u, Ds, f in (("aaaa", "aaaa", D[0], 1.0), ("abab", "abba", D[1], 2.0), ("bbbb", "bbbb", D[2], 1.0)):
        Y = f * _con("ijpq,klpq->ijkl", Ds, W[t])
        P = B[t] - B[u].permute(0, 1, 3, 2)                                    # B^{ij}_{kl} - B^{ij}_{lk}
        Pt = B[t].permute(2, 3, 0, 1) - B[u].permute(3, 2, 0, 1)               # B^{kl}_{ij} - B^{kl}_{ji}
        out.append(4.0 * (Y - s * Y.permute(2, 3, 0, 1)) - 12.0 * P + 12.0 * s * Pt)
    return tuple(out)


def _sum_so(X, Y):
    return (X[0] * Y[0]).sum() + (X[2] * Y[2]).sum() + 4.0 * (X[1] * Y[1]).sum()


def _exact_residual(K, D, case):
    A = _exact_G(tuple(0.5 * k for k in K), D, case, 1.0)
    return A, _sum_so(A, A)


def _exact_U(A, D, case):
    return tuple(0.5 * x for x in _exact_G(A, D, case, -1.0))


def _line_search(f0, f1, f2, e0):
    if abs(f1 - f0) <= 1e-10 * f0 and abs(f2 - f0) <= 1e-10 * f0:
        return 0.25 * e0
    c = (f0 - 2.0 * f1 + f2) / (2.0 * e0 * e0)
    if c > 0.0:
        x = -((f1 - f0) / e0 - c * e0) / (2.0 * c)
        return min(max(x, 0.25 * e0), 2.0 * e0)
    return e0 if f1 <= f2 else 2.0 * e0


def _exact_drive(K, D, case):
    """run_until_stop: steps with its stopping rule."""
    E, n2, eps, e0 = [float(_sum_so(K, D))], [], [], case["eps"]
    Ds, acc = [D], None
    for k in range(case["cap"]):
        A, f0 = _exact_residual(K, D, case)
        U = _exact_U(A, D, case)
        e = case["eps"]
        if case["ls"]:
            f = [float(_exact_residual(K, tuple(d + t * e0 * u for d, u in zip(D, U)), case)[1]) for t in (1.0, 2.0)]
            e = e0 = _line_search(float(f0), f[0], f[1], e0)
        D = tuple(d + e * u for d, u in zip(D, U))
        Ds.append(D)
        E.append(float(_sum_so(K, D)))
        n2.append(float(f0))
        eps.append(e)
        if k >= 1 and n2[k] > n2[k - 1] * (1.0 + 1e-10):
            acc = k - 1
        elif E[k + 1] > E[k] + 1e-12 * abs(E[k]):
            acc = k
        elif abs(E[k + 1] - E[k]) < 1e-6:
            acc = k + 1
        if acc is not None:
            break
        Ds = Ds[-2:]
    last = len(E) - 1
    acc = last if acc is None else acc
    return dict(E=np.array(E), norm2=np.array(n2), eps=np.array(eps), E_stop=E[acc], D=Ds[acc - last - 1])


def _exact_steps(K, D, case):
    for _ in range(case["nsteps"]):
        A, n2 = _exact_residual(K, D, case)
        D = tuple(d + case["eps"] * u for d, u in zip(D, _exact_U(A, D, case)))
    return D, _sum_so(K, D), n2


def _exact_adjoint(h, V, D, case):
    h, V = h.requires_grad_(True), V.requires_grad_(True)
    D0 = tuple(d.requires_grad_(True) for d in D)
    K = _exact_K(h, V, case["n"])
    D, E, _ = _exact_steps(K, D0, case)
    f = E + 0.01 * _exact_residual(K, D, case)[1]
    gh, gV, aa, ab, bb = torch.autograd.grad(f, (h, V) + D0)
    gV = 0.5 * (gV + gV.permute(1, 0, 2, 3))       # (pq|rs) symmetries, then those of a 2-RDM
    gV = 0.5 * (gV + gV.permute(0, 1, 3, 2))
    gV = 0.5 * (gV + gV.permute(2, 3, 0, 1))

    def pair(x, same):
        if same:
            x = 0.5 * (x - x.permute(1, 0, 2, 3))
            x = 0.5 * (x - x.permute(0, 1, 3, 2))
        return 0.5 * (x + x.permute(2, 3, 0, 1))

    return dict(dh=0.5 * (gh + gh.T), dV=gV, dD=(pair(aa, True), pair(ab, False), pair(bb, True)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        E, n2, D = [], [], []
        for i, inst in enumerate(_instances(case)):
            h, V, d = _problem(inst, seed + 7919 * i)
            d, e, n = _exact_steps(_exact_K(h, V, inst["n"]), d, dict(inst, nsteps=case["nsteps"], eps=case["eps"]))
            E.append(float(e))
            n2.append(float(n))
            D.append(d)
        return dict(E=np.array(E), norm2=np.array(n2), D=D)
    h, V, D = _problem(case, seed)
    if kind == "adjoint":
        if case["prec"] == "bf16x3":   # the gradient along that precision's own trajectory: no such value
            return None
        return _exact_adjoint(h, V, D, case)
    K = _exact_K(h, V, case["n"])
    if kind == "drive":
        return _exact_drive(K, D, case)
    if kind == "residual":
        A, n2 = _exact_residual(K, D, case)
        return dict(A=A, norm2=n2.reshape(1))
    D, E, n2 = _exact_steps(K, D, case)
    eps = torch.full((1,), case["eps"], dtype=F64, device=DEV)
    return dict(D=D, E=E.reshape(1), norm2=n2.reshape(1), eps=eps)
