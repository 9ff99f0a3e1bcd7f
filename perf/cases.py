"""The work a program has this library do, as cases that can be timed.

Three kinds of pass, each through the public Python entry points:

* ``propagate``: one RT-CC3 (or RT-CCSD) trajectory piece: upload the state of
  every field slot, ``nsteps`` RK4 steps, read the dipoles, the energies and the
  state back (the pattern of a finite-field or real-time property run);
* ``residuals``: one evaluation of all residuals, the energy and the dipole at
  given amplitudes (one RK4 stage; what a ground-state solver or an integrator
  of the user's own calls);
* ``triples``: the triples map and its vector-Jacobian product through
  ``TriplesResidual`` on device tensors (a differentiable block of a user's
  torch program).

Sizes follow the (H2O)n-like systems of ``synth.WATER_SIZES`` (nocc 5n, nvir
19n) and odd, ragged ones between nocc 3 and 20.  The FP64 form is the
library's default; the complex64-graph forms (FP32, split TF32, BF16 triples)
hand back what they computed in single precision, so their results are kept
in complex64, which is what such a program stores.

The start amplitudes are first-order ground-state amplitudes of the drawn
system plus a small complex part (a propagated state).
"""
import math

import numpy as np
import torch

from paper_2407_18947_gb300 import synth
from paper_2407_18947_gb300.api import FIELD_COS, FIELD_STATIC, RTCC3
from paper_2407_18947_gb300.autograd import TriplesResidual

PRECISION = {"fp64": 0, "fp32": 1, "tf32": 2, "bf16": 3}
H = 0.01  # RK4 step (au)
TIME = 0.3  # time of single evaluations (au)


def _case(name, kind, nocc, nvir, precision, **more):
    c = {"kind": kind, "nocc": nocc, "nvir": nvir, "precision": precision, "field": "static",
         "amplitude": 0.002, "slots": 1, "nsteps": 1, "triples": True, "chunk": 0}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest differentiable block: launches and host latency
        _case("triples_3x8_fp64", "triples", 3, 8, "fp64"),
        # the water-monomer-like system in the default FP64 form: ten RK4 steps
        # in a static field
        _case("propagate_5x19_fp64", "propagate", 5, 19, "fp64", nsteps=10),
        # finite-field set for polarisabilities: seven static fields in one
        # context, complex64 graph
        _case("fields7_5x19_tf32", "propagate", 5, 19, "tf32", slots=7, nsteps=5, amplitude=0.001),
        # one FP64 stage of a ragged system (a user's own integrator)
        _case("residuals_7x23_fp64", "residuals", 7, 23, "fp64"),
        # forward and reverse of the triples block in FP64, ragged
        _case("triples_9x31_fp64", "triples", 9, 31, "fp64", field="cos", amplitude=0.001),
        # RT-CCSD (triples off), the comparison mode, ragged
        _case("ccsd_11x41_fp64", "residuals", 11, 41, "fp64", triples=False),
        # one stage without tensor cores in the triples
        _case("residuals_8x27_fp32", "residuals", 8, 27, "fp32", field="cos", amplitude=0.001),
        # the water-dimer-like flagship: RK4 steps in an oscillating field, split TF32
        _case("propagate_10x38_tf32", "propagate", 10, 38, "tf32", field="cos", amplitude=0.001,
              nsteps=2),
        # the same with BF16 triples operands
        _case("propagate_10x38_bf16", "propagate", 10, 38, "bf16", field="cos", amplitude=0.001),
        # the plain FP64 form the reduced ones are compared with, at dimer size
        _case("residuals_10x38_fp64", "residuals", 10, 38, "fp64", field="cos", amplitude=0.001),
        # water-trimer size, triples blocked by occupied slabs (never stored)
        _case("residuals_15x57_tf32", "residuals", 15, 57, "tf32", chunk=5),
        # the largest: forward and reverse triples at water-tetramer size, blocked
        _case("triples_20x76_tf32", "triples", 20, 76, "tf32", chunk=2),
    ]


def draw(rng):
    kind = rng.choice(["propagate", "residuals", "residuals", "triples", "triples"])
    precision = rng.choice(["fp64", "fp64", "tf32", "tf32", "fp32", "bf16"])
    top = {"fp64": 10, "fp32": 10, "bf16": 11, "tf32": 14}[precision]
    if kind == "propagate":
        top = min(top, 8 if precision == "fp64" else 9)
    nocc = int(round(math.exp(rng.uniform(math.log(3), math.log(top)))))
    nvir = int(round(nocc * rng.uniform(2.6, 4.0)))
    chunk = 0
    if nocc >= 11:  # beyond dimer size the triples are blocked
        chunk = rng.randint(2, 5)
    return _case(None, kind, nocc, nvir, precision, field=rng.choice(["static", "cos"]),
                 amplitude=rng.choice([0.0005, 0.001, 0.002]),
                 slots=rng.choice([1, 2, 3]) if kind == "propagate" and nocc <= 6 else 1,
                 nsteps=rng.randint(1, 3) if kind == "propagate" else 1,
                 triples=(rng.random() < 0.85) if kind == "residuals" else True, chunk=chunk)


def _system(case, seed):
    return synth.make_system(case["nocc"], case["nvir"], seed=10_000 + int(seed))


def _amplitudes(s, seed):
    """First-order ground-state amplitudes plus a small complex part."""
    o = s.nocc
    eo, ev = s.eps[:o], s.eps[o:]
    lov = s.Lfac[:, :o, o:].reshape(s.naux, -1)
    g = (lov.T @ lov).reshape(o, s.nvir, o, s.nvir).transpose(0, 2, 1, 3)
    d = (ev[None, None, :, None] + ev[None, None, None, :]
         - eo[:, None, None, None] - eo[None, :, None, None])
    t2 = -g / d
    rng = np.random.Generator(np.random.PCG64(int(seed) + 77))

    def noise(shape, scale):
        return scale * (rng.standard_normal(shape) + 1j * rng.standard_normal(shape))

    def pair(x):
        return 0.5 * (x + x.transpose(1, 0, 3, 2))

    t1 = noise((o, s.nvir), 2e-3)
    l1 = noise((o, s.nvir), 4e-3)
    l2 = 2.0 * (2.0 * t2 - t2.transpose(0, 1, 3, 2))
    return (t1, t2 + pair(noise(t2.shape, 5e-4)), l1, l2 + pair(noise(t2.shape, 1e-3)))


def _fields(case):
    """(kind, amplitude, omega) of every slot: static sets are 0, +-A, +-2A, ..."""
    a = case["amplitude"]
    if case["field"] == "cos":
        return [(FIELD_COS, a * (1 + b), 0.0656) for b in range(case["slots"])]
    if case["slots"] == 1:
        return [(FIELD_STATIC, a, 0.0)]
    return [(FIELD_STATIC, a * ((b + 1) // 2) * (1 if b % 2 else -1), 0.0)
            for b in range(case["slots"])]


def prepare(case, seed):
    s = _system(case, seed)
    eng = RTCC3(s.nocc, s.nvir, nbatch=case["slots"], precision=PRECISION[case["precision"]],
                triples=bool(case["triples"]), triples_chunk=case["chunk"],
                storage_c64=case["slots"] > 1 and case["precision"] != "fp64")
    eng.set_hamiltonian(s.eps, s.Lfac, s.dipole)
    for b, (kind, amp, om) in enumerate(_fields(case)):
        eng.set_field(b, kind, amp, omega=om, direction=(0.0, 0.0, 1.0))
    amps = _amplitudes(s, seed)
    state = {"eng": eng, "case": case, "amps": amps}
    if case["kind"] == "residuals":
        eng.set_amplitudes(0, *amps)
    elif case["kind"] == "triples":
        state["dev"] = [torch.from_numpy(np.ascontiguousarray(x, dtype=np.complex128)).cuda()
                        for x in amps]
    return state


def run(state):
    eng, case = state["eng"], state["case"]
    keep = torch.complex128 if case["precision"] == "fp64" else torch.complex64
    npkeep = np.complex128 if case["precision"] == "fp64" else np.complex64
    if case["kind"] == "triples":
        t1, t2, u1, u2 = state["dev"]
        t1 = t1.detach().requires_grad_(True)
        t2 = t2.detach().requires_grad_(True)
        x1, x2 = TriplesResidual.apply(t1, t2, eng, 0, TIME)
        g1, g2 = torch.autograd.grad([x1, x2], [t1, t2], [u1, u2])
        return {"x1": x1.detach().to(keep), "x2": x2.detach().to(keep), "g1": g1.to(keep),
                "g2": g2.to(keep)}
    if case["kind"] == "residuals":
        r = eng.compute_residuals(0, TIME)
        out = {k: r[k].astype(npkeep) for k in ("r_t1", "r_t2", "r_l1", "r_l2", "dipole")}
        out["energy"] = np.asarray(r["energy"]).astype(npkeep)
        return out
    eng.set_time(0.0)
    for b in range(case["slots"]):
        eng.set_amplitudes(b, *state["amps"])
    dip, en = eng.propagate_rk4_chunk(H, case["nsteps"])
    out = {"dipole": dip.astype(npkeep), "energy": en.astype(npkeep)}
    for b in range(case["slots"]):
        for k, x in zip(("t1", "t2", "l1", "l2"), eng.get_amplitudes(b)):
            out[f"{k}_{b}"] = x.astype(npkeep)
    return out


# ---- what a pass cannot do without ---------------------------------------------

def _stage_macs(o, v, naux, triples):
    """Complex multiply-adds of one stage with its reverse pass (each product
    of the forward pass has two adjoints)."""
    n = o + v
    dress = 2.0 * naux * n ** 3 + naux * n ** 4
    ccsd = o * o * v ** 4 + o ** 4 * v * v * 2 + o ** 3 * v ** 3 * 5 + o * o * v ** 3 * 4
    m = 3.0 * (dress + ccsd)
    if triples:
        m += _triples_macs(o, v, 1, 2)
    return m


def _triples_macs(o, v, fwd, rev):
    t = float(o) ** 3 * float(v) ** 3
    # build over (e | l) and m, back-contractions over e and m; the field-coupling slot
    # densities belong to the reverse pass
    return t * ((v + 2 * o) + (v + o) + 4) * (fwd + rev) + (t * (v + o) if rev else 0.0)


def work(case):
    o, v = case["nocc"], case["nvir"]
    naux, n = 3 * (o + v), o + v
    amps = 16.0 * (o * v + o * o * v * v)
    ham = 8.0 * (naux * n * n + 4 * n * n)
    if case["kind"] == "triples":
        # forward, then the reverse (which needs the forward's values again)
        macs = (2 * (2.0 * naux * n ** 3 + naux * n ** 4) + _triples_macs(o, v, 1, 2))
        return {"bytes": ham + 6 * amps, "flops": 8.0 * macs}
    if case["kind"] == "residuals":
        return {"bytes": ham + 4 * amps, "flops": 8.0 * _stage_macs(o, v, naux, case["triples"])}
    k = case["slots"] * case["nsteps"] * 4
    return {"bytes": ham + 4 * amps * case["slots"],
            "flops": 8.0 * k * _stage_macs(o, v, naux, case["triples"])}


# ---- the same in 64 bits with plain torch --------------------------------------

_CD = torch.complex128


def _es(spec, *xs):
    return torch.einsum(spec, *xs)


class _SolveT3(torch.autograd.Function):
    """Derivative of A^-1 at r = 0 (A = D3 + the field's slot operator): the
    forward value is zero, the reverse solves the transposed equation."""

    @staticmethod
    def forward(ctx, r, d3, woo, wvv):
        ctx.save_for_backward(d3, woo, wvv)
        return torch.zeros_like(r)

    @staticmethod
    def backward(ctx, g):
        d3, woo, wvv = ctx.saved_tensors
        # torch's complex convention: grad_in = (A^-T)^* grad_out
        return _fixed_point(g, d3, woo.conj().T.contiguous(), wvv.conj().T.contiguous()), None, None, None


def _slot(woo, wvv, t):
    return (_es("ad,ijkdbc->ijkabc", wvv, t) + _es("bd,ijkadc->ijkabc", wvv, t)
            + _es("cd,ijkabd->ijkabc", wvv, t) - _es("li,ljkabc->ijkabc", woo, t)
            - _es("lj,ilkabc->ijkabc", woo, t) - _es("lk,ijlabc->ijkabc", woo, t))


def _fixed_point(rhs, d3, woo, wvv):
    t = rhs / d3
    for _ in range(60):
        new = (rhs - _slot(woo, wvv, t)) / d3
        far, big = float((new - t).abs().max()), float(new.abs().max())
        t = new
        if far <= 1e-16 * big:
            break
    return t


class _Exact:
    def __init__(self, s, dev):
        self.o, self.dev = s.nocc, dev
        f = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), device=dev).to(_CD)  # noqa: E731
        self.eps, self.L, self.mu = f(s.eps), f(s.Lfac), f(s.dipole)
        o, n = self.o, self.eps.numel()
        self.n, self.v = n, n - o
        lk = _es("Pkk->P", self.L[:, :o, :o])
        j = _es("Ppq,P->pq", self.L, lk)
        k = _es("Ppk,Pkq->pq", self.L[:, :, :o], self.L[:, :o, :])
        self.h = torch.diag(self.eps) - 2 * j + k
        eo, ev = self.eps[:o], self.eps[o:]
        occ = eo[:, None, None] + eo[None, :, None] + eo[None, None, :]
        vir = ev[:, None, None] + ev[None, :, None] + ev[None, None, :]
        self.occ, self.vir = occ, vir

    def d3(self):
        return self.vir[None, None, None] - self.occ[:, :, :, None, None, None]

    def dress(self, t1, w):
        o, v, n = self.o, self.v, self.n
        z = torch.zeros
        tau = torch.cat([z(o, n, dtype=_CD, device=self.dev),
                         torch.cat([t1.T, z(v, v, dtype=_CD, device=self.dev)], 1)], 0)
        eye = torch.eye(n, dtype=_CD, device=self.dev)
        x, y = eye - tau, eye + tau
        lt = _es("pr,Prs,sq->Ppq", x, self.L, y)
        g = _es("Ppq,Prs->pqrs", lt, lt)
        f = x @ (self.h + w) @ y + 2 * _es("pqkk->pq", g[:, :, :o, :o]) \
            - _es("pkkq->pq", g[:, :o, :o, :])
        return g, f, x @ w @ y

    def ccsd(self, g, f, t):
        o = self.o
        O, V = slice(0, o), slice(o, self.n)
        u = 2 * t - t.transpose(2, 3)
        gov = g[O, V, O, V]
        r1 = _es("kicd,adkc->ia", u, g[V, V, O, V]) - _es("klac,kilc->ia", u, g[O, O, O, V]) \
            + _es("ikac,kc->ia", u, f[O, V]) + f[V, O].T
        w = g[O, O, O, O] + _es("ijcd,kcld->kilj", t, gov)
        r2 = _es("aibj->ijab", g[V, O, V, O]) + _es("ijcd,acbd->ijab", t, g[V, V, V, V]) \
            + _es("klab,kilj->ijab", t, w)
        xc = g[O, O, V, V] - 0.5 * _es("liad,kdlc->kiac", t, gov)
        s = -0.5 * _es("kjbc,kiac->ijab", t, xc) - _es("kibc,kjac->ijab", t, xc)
        lov = 2 * gov - _es("lckd->ldkc", gov)
        xd = _es("aikc->iakc", 2 * g[V, O, O, V] - _es("acki->aikc", g[V, V, O, O])) \
            + 0.5 * _es("ilad,ldkc->iakc", u, lov)
        s = s + 0.5 * _es("jkbc,iakc->ijab", u, xd)
        fvv = f[V, V] - _es("klbd,ldkc->bc", u, gov)
        foo = f[O, O] + _es("ljcd,kdlc->kj", u, gov)
        s = s + _es("ijac,bc->ijab", t, fvv) - _es("ikab,kj->ijab", t, foo)
        return r1, r2 + s + s.permute(1, 0, 3, 2)

    def triples(self, g, f, wt, t):
        o = self.o
        O, V = slice(0, o), slice(o, self.n)
        z = _es("ijae,ckbe->ijkabc", t, g[V, O, V, V]) - _es("imab,mjck->ijkabc", t, g[O, O, V, O]) \
            - _es("lija,klcb->ijkabc", _es("ld,ijad->lija", wt[O, V], t), t)
        rhs = -sum(z.permute(*p, *(3 + k for k in p))
                   for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)))
        d3, woo, wvv = self.d3(), wt[O, O], wt[V, V]
        with torch.no_grad():
            t3 = _fixed_point(rhs, d3, woo, wvv)
        if rhs.requires_grad:
            r = rhs - d3 * t3 - _slot(woo, wvv, t3)
            t3 = t3 + _SolveT3.apply(r, d3, woo.detach(), wvv.detach())
        gov = g[O, V, O, V]
        dd = t3 - t3.permute(0, 1, 2, 5, 4, 3)
        x1 = _es("ijkabc,jkbc->ia", dd, 2 * _es("jbkc->jkbc", gov) - _es("jckb->jkbc", gov))
        s = _es("ijkabc,kc->ijab", dd, f[O, V])
        ub = 2 * t3 - t3.permute(0, 1, 2, 3, 5, 4) - t3.permute(0, 1, 2, 5, 4, 3)
        s = s + _es("ijkcbe,acke->ijab", ub, g[V, V, O, V])
        uc = 2 * t3 - t3.permute(0, 1, 2, 4, 3, 5) - t3.permute(0, 1, 2, 5, 4, 3)
        s = s - _es("mjkcba,kimc->ijab", uc, g[O, O, O, V])
        return x1, s + s.permute(1, 0, 3, 2)

    def field(self, case, b, t):
        kind, amp, om = _fields(case)[b]
        e = amp * (math.cos(om * t) if kind == FIELD_COS else 1.0)
        return -e * self.mu[2]

    def triples_map(self, t1, t2, w):
        g, f, wt = self.dress(t1, w)
        return self.triples(g, f, wt, t2)

    def stage(self, amps, w, triples):
        t1, t2, w = (x.detach().clone().requires_grad_(True) for x in (amps[0], amps[1], w))
        o = self.o
        with torch.enable_grad():
            g, f, wt = self.dress(t1, w)
            r1, r2 = self.ccsd(g, f, t2)
            if triples:
                x1, x2 = self.triples(g, f, wt, t2)
                r1, r2 = r1 + x1, r2 + x2
            lov = _es("Pia,Pjb->iajb", self.L[:, :o, o:], self.L[:, :o, o:])
            lov = 2 * lov - _es("ibja->iajb", lov)
            e = 2 * _es("ii->", w[:o, :o]) + 2 * (w[:o, o:] * t1).sum() \
                + _es("iajb,ijab->", lov, t2 + _es("ia,jb->ijab", t1, t1))
            lag = e + (amps[2] * r1).sum() + 0.5 * (amps[3] * r2).sum()
            g1, g2, gw = (x.conj().resolve_conj() for x in torch.autograd.grad(lag.real, [t1, t2, w]))
        dip = _es("pq,xpq->x", gw, self.mu)
        return (r1.detach(), r2.detach(), g1, g2 + g2.permute(1, 0, 3, 2)), dip, e.detach()


def exact(case, seed):
    o, v = case["nocc"], case["nvir"]
    stages = {"propagate": 4 * case["nsteps"] * case["slots"], "residuals": 1, "triples": 1}[case["kind"]]
    if case["triples"] and ((o * v) ** 3 * (20 * (o + v)) * 8.0 * stages > 1.5e13
                            or (o * v) ** 3 > 3e8):
        return None  # about 20 seconds of 64-bit arithmetic, or 150 GB of 64-bit tensors
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    s = _system(case, seed)
    x = _Exact(s, dev)
    amps = [torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).to(dev)
            for a in _amplitudes(s, seed)]
    if case["kind"] == "triples":
        t1, t2 = (a.clone().requires_grad_(True) for a in amps[:2])
        x1, x2 = x.triples_map(t1, t2, x.field(case, 0, TIME))
        g1, g2 = torch.autograd.grad([x1, x2], [t1, t2], [amps[2], amps[3]])
        return {"x1": x1.detach(), "x2": x2.detach(), "g1": g1, "g2": g2}
    if case["kind"] == "residuals":
        r, dip, e = x.stage(amps, x.field(case, 0, TIME), case["triples"])
        return {"r_t1": r[0], "r_t2": r[1], "r_l1": r[2], "r_l2": r[3], "dipole": dip, "energy": e}
    out, dips, ens = {}, [], []
    sign = (-1j, -1j, 1j, 1j)
    for b in range(case["slots"]):
        y, dip_b, en_b = amps, [], []
        for n in range(case["nsteps"]):
            k, acc = None, [torch.zeros_like(a) for a in y]
            for c, wgt in ((0.0, 1.0), (0.5, 2.0), (0.5, 2.0), (1.0, 1.0)):
                at = y if k is None else [a + c * H * d for a, d in zip(y, k)]
                r, dip, e = x.stage(at, x.field(case, b, (n + c) * H), case["triples"])
                if c == 0.0:
                    dip_b.append(dip)
                    en_b.append(e)
                k = [sg * d for sg, d in zip(sign, r)]
                acc = [a + wgt * d for a, d in zip(acc, k)]
            y = [a + (H / 6.0) * d for a, d in zip(y, acc)]
        dips.append(torch.stack(dip_b))
        ens.append(torch.stack(en_b))
        for name, a in zip(("t1", "t2", "l1", "l2"), y):
            out[f"{name}_{b}"] = a
    out["dipole"], out["energy"] = torch.stack(dips), torch.stack(ens)
    return out
