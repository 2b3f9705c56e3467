"""Performance cases: the work a user of the framework has it do, through its public Python entry points.

A case is a dict of plain values; ``prepare`` builds what a program holds before the call (inputs, contexts
with their integrals and plans), ``run`` is one pass, ``exact`` the same results from plain dense torch in
64 bits (its own integrals from the published recipe, the amplitude equations on full arrays).

Kinds:
  ccsd    restart from given amplitudes, a few CCSD iterations, amplitudes and energy back
  batch   many small Hamiltonians in one context: learned guess, a few iterations, everything back
  t3      the (T) correction of the amplitudes a context holds
  solve   a whole calculation: context, integrals, convergence, the (0h,1p) sector
  zgemm   one complex matrix product
  train   epochs of the learned guess on converged amplitudes
"""
import itertools
import math

import numpy as np
import torch

from paper_2004_03682_gb300 import expgb
from paper_2004_03682_gb300 import synthetic as syn

DEV = "cuda"


def listed():
    return [
        # the smallest calculation in plain FP64: no symmetry, one instance; launches and FP64 rate
        dict(name="ccsd_c1_o10_v40_fp64", kind="ccsd", o=10, v=40, g=1, prec="fp64", s=5, sm=0, real=False, iters=2, shift=0.0),
        # the same Hamiltonian on the emulated path: latency of a short dependent chain
        dict(name="ccsd_c1_o10_v40_emu", kind="ccsd", o=10, v=40, g=1, prec="emu", s=5, sm=0, real=False, iters=4, shift=0.0),
        # ragged sizes: odd counts, an odd group, six slices everywhere
        dict(name="ccsd_z3_o23_v117_s6", kind="ccsd", o=23, v=117, g=3, prec="emu", s=6, sm=0, real=False, iters=3, shift=8.0),
        # a real Hamiltonian (real double groups) in real arithmetic
        dict(name="ccsd_z4_o32_v160_real", kind="ccsd", o=32, v=160, g=4, prec="emu", s=6, sm=5, real=True, iters=2, shift=8.0),
        # the symmetry-blocked workload
        dict(name="ccsd_z8_o40_v200_s5", kind="ccsd", o=40, v=200, g=8, prec="emu", s=5, sm=0, real=False, iters=2, shift=8.0),
        # the largest: five slices for the ladder and ring products, six for the others
        dict(name="ccsd_z8_o48_v300_s65", kind="ccsd", o=48, v=300, g=8, prec="emu", s=6, sm=5, real=False, iters=2, shift=32.0),
        # many small Hamiltonians solved together from the learned guess
        dict(name="batch_o10_v40_x64", kind="batch", o=10, v=40, n=64, s=5, iters=5),
        # (T), a mid-sized and a large one
        dict(name="t3_z4_o18_v72", kind="t3", o=18, v=72, g=4, prec="emu", s=5),
        dict(name="t3_z8_o40_v200", kind="t3", o=40, v=200, g=8, prec="emu", s=5),
        # a whole small calculation with the Fock-space sector, set-up included
        dict(name="solve_z4_o12_v48_a4", kind="solve", o=12, v=48, g=4, active=4, s=6),
        # one large complex product outside any context
        dict(name="zgemm_2048_s6", kind="zgemm", m=2048, n=2048, k=2048, prec="emu", s=6),
        # training of the learned guess
        dict(name="train_o10_v40_x16", kind="train", o=10, v=40, n=16, epochs=2, batch=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ccsd", "ccsd", "ccsd", "ccsd", "batch", "t3", "t3", "solve", "zgemm", "zgemm", "train"])
    if kind == "ccsd":
        while True:
            prec = rng.choice(["emu", "emu", "emu", "fp64"])
            o, v, g = _log(rng, 8, 44), _log(rng, 30, 280), rng.choice([1, 2, 3, 4, 5, 8, 16])
            most = _ccsd_macs(48, 300, 8) / (1 if prec == "emu" else 40)
            if v >= 2 * o and _ccsd_macs(o, v, g) <= 0.7 * most and _ccsd_bytes(o, v, g) <= 0.5 * _ccsd_bytes(48, 300, 8):
                break
        s = rng.choice([4, 5, 5, 6, 6])
        return dict(kind=kind, o=o, v=v, g=g, prec=prec, s=s, sm=5 if s == 6 and rng.random() < 0.5 else 0,
                    real=prec == "emu" and rng.random() < 0.25, iters=rng.choice([1, 2, 3]), shift=8.0)
    if kind == "batch":
        return dict(kind=kind, o=rng.randint(6, 12), v=rng.randint(20, 44), n=_log(rng, 4, 96), s=rng.choice([5, 6]), iters=rng.choice([2, 3, 5]))
    if kind == "t3":
        g = rng.choice([1, 2, 4, 5, 8])
        while True:
            o, v = _log(rng, 6, 36), _log(rng, 24, 180)
            if v >= 2 * o and _t3_macs(o, v, g) <= 0.4 * _t3_macs(40, 200, 8):
                return dict(kind=kind, o=o, v=v, g=g, prec="emu", s=rng.choice([5, 6]))
    if kind == "solve":
        return dict(kind=kind, o=rng.randint(6, 16), v=rng.randint(24, 64), g=rng.choice([1, 2, 4]), active=rng.randint(1, 4), s=rng.choice([5, 6]))
    if kind == "zgemm":
        prec = rng.choice(["emu", "emu", "emu", "fp64", "ds"])
        while True:
            m, n = _log(rng, 16, 6000), _log(rng, 16, 6000)
            k = rng.randint(1, 16) if prec == "ds" else _log(rng, 16, 12000)
            if m * n * k <= 2048 ** 3 / (1 if prec != "fp64" else 60):
                return dict(kind=kind, m=m, n=n, k=k, prec=prec, s=rng.choice([3, 4, 5, 6]))
    return dict(kind="train", o=rng.randint(6, 10), v=rng.randint(24, 40), n=rng.randint(4, 16), epochs=rng.choice([1, 2, 4]), batch=rng.choice([4096, 16384, 65536]))


# ---------------------------------------------------------------------------------------------------------
# inputs


def _problem(o, v, g, seed, k=0, scale=1.0, active=0):
    """Member k of a seeded family of Hamiltonians: the irrep partition belongs to the sizes (as a molecule's
    does), the orbital energies and the integrals' seed to the seed.  The `active` lowest virtual spinors lie
    1 hartree below the others: a model space without intruder states."""
    part = syn.make_problem(2001, o, v, g)
    rng = np.random.default_rng([seed, k, 17])
    eo = np.concatenate([np.sort(rng.uniform(-2.0, -0.5, int(c))) for c in part.irrep_occ])
    ev = np.concatenate([np.sort(rng.uniform(0.2, 5.0, int(c))) for c in part.irrep_virt])
    if active:
        ev = ev + 1.0 * (ev > np.sort(ev)[active - 1])
    return syn.Problem(int(rng.integers(1, 2 ** 48)), o, v, g, part.irrep_occ, part.irrep_virt, eo, ev, scale)


def _amplitudes(p, seed):
    """Amplitudes with the structure and the decay of converged ones: antisymmetric, symmetry-allowed, Gaussian
    over the energy denominators, at most 0.01 (t1) and 0.05 (t2)."""
    gen = torch.Generator(device=DEV).manual_seed(seed * 7919 + 5)
    o, v = p.n_occ, p.n_virt
    irr = torch.as_tensor(p.irrep_of, device=DEV)
    go, gv = irr[:o], irr[o:]
    eo, ev = torch.as_tensor(p.eps_occ, device=DEV), torch.as_tensor(p.eps_virt, device=DEV)
    t1 = torch.complex(*(torch.randn(o, v, generator=gen, device=DEV, dtype=torch.float64) for _ in range(2)))
    t1 = t1 * (go[:, None] == gv[None, :]) / (eo[:, None] - ev[None, :])
    t1 *= 0.01 / max(float(t1.abs().max()), 1e-300)
    t2 = torch.empty(o, o, v, v, dtype=torch.complex128, device=DEV)
    d = eo[:, None, None] - ev[None, :, None] - ev[None, None, :]
    for i in range(o):  # one row of pairs at a time: the large cases do not fit twice
        x = torch.complex(*(torch.randn(i, v, v, generator=gen, device=DEV, dtype=torch.float64) for _ in range(2)))
        x = (x - x.transpose(1, 2)) / (d[:i] + eo[i])
        x *= ((go[:i, None, None] + go[i] - gv[None, :, None] - gv[None, None, :]) % p.G) == 0
        t2[i, :i], t2[:i, i], t2[i, i] = x, -x, 0
    t2 *= 0.05 / max(max(float(t2[i].abs().max()) for i in range(o)), 1e-300)
    return t1, t2


def _real(t1, t2):
    return t1.real.to(torch.complex128), t2.real.to(torch.complex128)


def _precision(c):
    return {"fp64": expgb.EXP_FP64, "emu": expgb.EXP_EMU_BF16, "ds": expgb.EXP_EMU_DS}[c["prec"]]


def _zgemm_inputs(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed * 7919 + 11)
    a, b = (torch.complex(*(torch.randn(x, y, generator=gen, device=DEV, dtype=torch.float64) for _ in range(2)))
            for x, y in ((c["m"], c["k"]), (c["k"], c["n"])))
    # rows and columns of unequal size, as integrals and amplitudes have them
    a *= torch.exp(2.0 * torch.randn(c["m"], 1, generator=gen, device=DEV, dtype=torch.float64))
    b *= torch.exp(2.0 * torch.randn(1, c["n"], generator=gen, device=DEV, dtype=torch.float64))
    return a, b


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "ccsd":
        p = _problem(c["o"], c["v"], c["g"], seed)
        t1, t2 = _amplitudes(p, seed)
        if c["real"]:
            t1, t2 = _real(t1, t2)
        ctx = expgb.from_problems([p], precision=_precision(c), n_slices=c["s"], n_slices_major=c["sm"], conv_tol=1e-30,
                                  max_iter=1 << 20, level_shift=c["shift"], real_arith=c["real"])
        ctx.init_integrals([p.seed])
        ctx.iterate(2)  # a program's first iterations: the plans and the iteration's graph
        return dict(c=c, ctx=ctx, t1=t1, t2=t2)
    if kind == "batch":
        probs = [_problem(c["o"], c["v"], 1, seed, k, 0.5 + (k % 8) / 8.0) for k in range(c["n"])]
        ctx = expgb.from_problems(probs, precision=expgb.EXP_EMU_BF16, n_slices=c["s"], conv_tol=1e-30, max_iter=1 << 20)
        ctx.init_integrals([p.seed for p in probs], scale_mult=[p.scale_mult for p in probs])
        ctx.iterate(2)
        return dict(c=c, ctx=ctx, mlp=expgb.Mlp(seed=seed, bf16=True))
    if kind == "t3":
        p = _problem(c["o"], c["v"], c["g"], seed)
        t1, t2 = _amplitudes(p, seed)
        ctx = expgb.from_problems([p], precision=_precision(c), n_slices=c["s"])
        ctx.init_integrals([p.seed])
        ctx.set_amplitudes(0, t1, t2)
        return dict(c=c, ctx=ctx)
    if kind == "solve":
        return dict(c=c, p=_problem(c["o"], c["v"], c["g"], seed, scale=0.4, active=c["active"]))
    if kind == "zgemm":
        a, b = _zgemm_inputs(c, seed)
        return dict(c=c, a=a, b=b)
    probs = [_problem(c["o"], c["v"], 1, seed, k, 0.4) for k in range(c["n"])]
    ctx = expgb.from_problems(probs, precision=expgb.EXP_EMU_BF16, conv_tol=1e-6, max_iter=200)
    ctx.init_integrals([p.seed for p in probs], scale_mult=[p.scale_mult for p in probs])
    ctx.iterate(200, raise_numeric=False)
    mlp = expgb.Mlp(seed=seed, bf16=True)
    mlp.add_training_data(ctx)
    ctx.close()
    return dict(c=c, mlp=mlp, start=mlp.params())


# ---------------------------------------------------------------------------------------------------------
# one pass


def _number(z):
    return np.array([z.real, z.imag])


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "ccsd":
        ctx = state["ctx"]
        ctx.set_amplitudes(0, state["t1"], state["t2"])
        recs, _, _ = ctx.iterate(c["iters"])
        t1, t2 = ctx.get_amplitudes(0)
        return dict(t1=t1, t2=t2, energy=_number(recs[-1]["e"]), max_dt=recs[-1]["max_dt"])
    if kind == "batch":
        ctx = state["ctx"]
        state["mlp"].apply(ctx)
        ctx.iterate(c["iters"])
        amps = [ctx.get_amplitudes(k) for k in range(c["n"])]
        return dict(t1=torch.stack([a for a, _ in amps]), t2=torch.stack([b for _, b in amps]),
                    energy=np.array([_number(ctx.energy(k)) for k in range(c["n"])]))
    if kind == "t3":
        e, _, per = state["ctx"].ccsd_t(per_triple=True)
        return dict(energy=_number(e), per_triple=per)
    if kind == "solve":
        p = state["p"]
        ctx = expgb.from_problems([p], precision=expgb.EXP_EMU_BF16, n_slices=c["s"], conv_tol=1e-10, max_iter=400,
                                  active=syn.active_virtuals(p, c["active"]), level_shift=2.0)
        ctx.init_integrals([p.seed], scale_mult=[p.scale_mult])
        ctx.iterate(400, raise_notconv=True)
        e = ctx.energy(0)
        heff, eig, _, _ = ctx.fs_sector_0h1p(0)
        ctx.close()
        return dict(energy=_number(e), heff=heff, eig=eig)
    if kind == "zgemm":
        return expgb.zgemm(state["a"], state["b"], precision=_precision(c), n_slices=c["s"])
    mlp = state["mlp"]
    mlp.params(set=state["start"])
    losses = mlp.train(c["epochs"], batch=c["batch"], lr=2e-3, seed=1)
    return dict(losses=losses, params=mlp.params())


# ---------------------------------------------------------------------------------------------------------
# work: complex multiply-adds count 8 flops; the sums over symmetry-allowed blocks as if irreps were even


def _ccsd_macs(o, v, g):
    pv, po = v * (v - 1) / 2, o * (o - 1) / 2
    ladder, hh, x = pv * pv * po, pv * po * po, o * v * pv * po
    ring = 2.0 * (o * v) ** 3
    o2v3 = 4.0 * o * o * v ** 3
    o3v2 = 5.0 * o ** 3 * v * v
    return (ladder + hh + x + ring + o2v3 + o3v2) / (g * g)


def _ccsd_bytes(o, v, g):
    """integrals once (pairs packed) and the amplitudes in and out"""
    pv, po = v * (v - 1) / 2, o * (o - 1) / 2
    return 16.0 * ((pv * pv / 2 + o * v * pv + po * pv + (o * v) ** 2 + o * v * po + po * po) / g + 2 * (o * v + o * o * v * v))


def _t3_macs(o, v, g):
    return o * (o - 1) * (o - 2) / 6 * 3 * (v + o) * v * (v * (v - 1) / 2) / (g * g)


def work(case):
    c, kind = case, case["kind"]
    if kind == "ccsd":
        per = 2.0 if c["real"] else 8.0
        return dict(bytes=_ccsd_bytes(c["o"], c["v"], c["g"]) * c["iters"], flops=per * _ccsd_macs(c["o"], c["v"], c["g"]) * c["iters"])
    if kind == "batch":
        return dict(bytes=_ccsd_bytes(c["o"], c["v"], 1) * c["iters"] * c["n"], flops=8.0 * _ccsd_macs(c["o"], c["v"], 1) * c["iters"] * c["n"])
    if kind == "t3":
        o, v, g = c["o"], c["v"], c["g"]
        return dict(bytes=16.0 * (o * v ** 3 / 2 + o * o * v * v + o ** 3 * v / 2) / g, flops=8.0 * _t3_macs(o, v, g))
    if kind == "solve":
        # about twenty iterations of each sector; the second carries the active spinors as further occupied ones
        o, v, g = c["o"] + c["active"], c["v"], c["g"]
        return dict(bytes=40 * _ccsd_bytes(o, v, g), flops=40 * 8.0 * _ccsd_macs(o, v, g))
    if kind == "zgemm":
        m, n, k = c["m"], c["n"], c["k"]
        return dict(bytes=16.0 * (m * k + k * n + m * n), flops=8.0 * m * n * k)
    n = c["n"] * (c["o"] * (c["o"] - 1) / 2) * (c["v"] * (c["v"] - 1) / 2)
    return dict(bytes=28.0 * n * c["epochs"], flops=6.0 * n * (3 * 128 + 128 * 128 + 256) * c["epochs"])


# ---------------------------------------------------------------------------------------------------------
# 64-bit results, dense


def _philox_normal(idx, seed):
    """A[idx]: Philox4x32-10 at counter (idx, 0, 0) and key seed, the Box-Muller pair of two 53-bit uniforms."""
    low = 0xFFFFFFFF
    x0, x1 = idx & low, (idx >> 32) & low
    x2, x3 = torch.zeros_like(x0), torch.zeros_like(x0)
    k0, k1 = seed & low, (seed >> 32) & low
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
        a, b = x0 * 0xD2511F53, x2 * 0xCD9E8D57  # wraps modulo 2^64
        x0, x1, x2, x3 = ((b >> 32) & low) ^ x1 ^ k0, b & low, ((a >> 32) & low) ^ x3 ^ k1, a & low
    u1 = ((((x1 << 32) | x0) >> 11) & ((1 << 53) - 1)).double().add_(0.5).mul_(2.0 ** -53)
    u2 = ((((x3 << 32) | x2) >> 11) & ((1 << 53) - 1)).double().add_(0.5).mul_(2.0 ** -53)
    rad, ang = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
    return torch.complex(rad * torch.cos(ang), rad * torch.sin(ang))


class _Hamiltonian:
    """Integrals <pq||rs> of the synthetic recipe on broadcastable global indices."""

    def __init__(self, p, real=False, scale=1.0):
        self.p, self.real, self.s, self.held = p, real, 1.0, {}
        self.irr = torch.as_tensor(p.irrep_of, device=DEV)
        self.o, self.n = p.n_occ, p.n
        self.O, self.V = torch.arange(self.o, device=DEV), torch.arange(self.o, self.n, device=DEV)
        self.eo, self.ev = torch.as_tensor(p.eps_occ, device=DEV), torch.as_tensor(p.eps_virt, device=DEV)
        self.D1 = self.eo[:, None] - self.ev
        self.D2 = self.eo[:, None, None, None] + self.eo[:, None, None] - self.ev[:, None] - self.ev
        v = self.fresh("vvoo").permute(2, 3, 0, 1)
        self.s = 0.05 / float((v.abs() / self.D2.abs()).max()) * scale

    def at(self, p, q, r, s):
        n = self.n
        A = lambda w, x, y, z: _philox_normal(((w * n + x) * n + y) * n + z, self.p.seed)  # noqa: E731
        v = A(p, q, r, s) - A(q, p, r, s) - A(p, q, s, r) + A(q, p, s, r)
        w = A(r, s, p, q) - A(s, r, p, q) - A(r, s, q, p) + A(s, r, q, p)
        v = 0.5 * (v + w.conj())
        if self.real:
            v = v.real.to(torch.complex128)
        ok = (self.irr[p] + self.irr[q] - self.irr[r] - self.irr[s]) % self.p.G == 0
        return v * ok * self.s

    def block(self, spec):
        if spec not in self.held:
            self.held[spec] = self.fresh(spec)
        return self.held[spec]

    def fresh(self, spec):
        i = [self.O if x == "o" else self.V for x in spec]
        out = torch.empty([len(x) for x in i], dtype=torch.complex128, device=DEV)
        for k, x in enumerate(i[0]):
            out[k] = self.at(x.view(1, 1, 1), i[1][:, None, None], i[2][:, None], i[3])
        return out

    def vvvv(self):
        """<ab||ef> for a<b, e<f"""
        if "vvvv" not in self.held:
            a, b = torch.triu_indices(len(self.V), len(self.V), 1, device=DEV) + self.o
            out = torch.empty(len(a), len(a), dtype=torch.complex128, device=DEV)
            step = max(1, (1 << 25) // max(len(a), 1))
            for r in range(0, len(a), step):
                out[r:r + step] = self.at(a[r:r + step, None], b[r:r + step, None], a, b)
            self.held["vvvv"] = out
        return self.held["vvvv"]


def _es(spec, a, b):
    """einsum of two operands as one matrix product"""
    i, out = spec.split("->")
    x, y = i.split(",")
    k = [q for q in x if q in y and q not in out]
    fx, fy = [q for q in x if q not in k], [q for q in y if q not in k]
    A = a.permute([x.index(q) for q in fx + k]).reshape(math.prod(a.shape[x.index(q)] for q in fx), -1)
    B = b.permute([y.index(q) for q in k + fy]).reshape(A.shape[1], -1)
    r = (A @ B).reshape([a.shape[x.index(q)] for q in fx] + [b.shape[y.index(q)] for q in fy])
    return r.permute([(fx + fy).index(q) for q in out])


def _tau(t1, t2, f=1.0):
    x = t1[:, None, :, None] * t1[None, :, None, :]
    return t2 + f * (x - x.transpose(2, 3))


def _rhs(h, t1, t2):
    """Right-hand sides of the spin-orbital CCSD equations (Stanton, Gauss, Watts and Bartlett, J. Chem. Phys. 94, 4334
    (1991)) for a diagonal Fock matrix, the W_abef products taken apart so that no v^4 intermediate is formed."""
    b = h.block
    o, v = t1.shape
    ta, tt = _tau(t1, t2), _tau(t1, t2, 0.5)
    Fae = _es("mf,mafe->ae", t1, b("ovvv")) - 0.5 * _es("mnaf,mnef->ae", tt, b("oovv"))
    Fmi = _es("ne,mnie->mi", t1, b("ooov")) + 0.5 * _es("inef,mnef->mi", tt, b("oovv"))
    Fme = _es("nf,mnef->me", t1, b("oovv"))
    w = _es("je,mnie->mnij", t1, b("ooov"))
    Wmn = b("oooo") + w - w.transpose(2, 3) + 0.5 * _es("ijef,mnef->mnij", ta, b("oovv"))  # with W_abef's tau term
    z = 0.5 * t2 + t1[:, None, :, None] * t1[None, :, None, :]
    Wr = (b("ovvo") + _es("jf,mbef->mbej", t1, b("ovvv")) - _es("nb,mnej->mbej", t1, b("oovo"))
          - _es("jnfb,mnef->mbej", z, b("oovv")))
    r1 = (_es("ie,ae->ia", t1, Fae) - _es("ma,mi->ia", t1, Fmi) + _es("imae,me->ia", t2, Fme)
          - _es("nf,naif->ia", t1, b("ovov")) - 0.5 * _es("imef,maef->ia", t2, b("ovvv"))
          - 0.5 * _es("mnae,nmei->ia", t2, b("oovo")))
    r2 = b("vvoo").permute(2, 3, 0, 1).clone()
    x = _es("ijae,be->ijab", t2, Fae - 0.5 * _es("mb,me->be", t1, Fme))
    r2 += x - x.transpose(2, 3)
    x = _es("imab,mj->ijab", t2, Fmi + 0.5 * _es("je,me->mj", t1, Fme))
    r2 -= x - x.transpose(0, 1)
    r2 += 0.5 * _es("mnab,mnij->ijab", ta, Wmn)
    pa, pb = torch.triu_indices(v, v, 1, device=DEV)
    pi, pj = torch.triu_indices(o, o, 1, device=DEV)
    lad = h.vvvv() @ ta[pi, pj][:, pa, pb].T  # (a<b, i<j)
    for (i, j, si), (a, e, sa) in itertools.product(((pi, pj, 1), (pj, pi, -1)), ((pa, pb, 1), (pb, pa, -1))):
        r2[i[:, None], j[:, None], a[None, :], e[None, :]] += si * sa * lad.T
    X = _es("ijef,maef->ijma", ta, b("ovvv"))  # -<am||ef> tau
    x = 0.5 * _es("mb,ijma->ijab", t1, X)
    r2 += x - x.transpose(2, 3)
    x = _es("imae,mbej->ijab", t2, Wr) - _es("ma,mbij->ijab", t1, _es("ie,mbej->mbij", t1, b("ovvo")))
    x = x - x.transpose(0, 1)
    r2 += x - x.transpose(2, 3)
    x = _es("ie,abej->ijab", t1, b("vvvo"))
    r2 += x - x.transpose(0, 1)
    x = _es("ma,mbij->ijab", t1, b("ovoo"))
    r2 -= x - x.transpose(2, 3)
    return r1, r2


def _energy(h, t1, t2):
    v = h.block("vvoo").permute(2, 3, 0, 1).conj()
    return complex(0.25 * (v * _tau(t1, t2)).sum())


def _iterate(h, t1, t2, iters, shift, tol=0.0):
    """Jacobi steps t <- t + (RHS - D t) / (D - shift) with Pulay DIIS(6) -> (t1, t2, E(t_new), max |t_new - t|)"""
    vecs, errs, e, mx = [], [], None, None
    for _ in range(iters):
        r1, r2 = _rhs(h, t1, t2)
        n1, n2 = (r1 - shift * t1) / (h.D1 - shift), (r2 - shift * t2) / (h.D2 - shift)
        err = torch.cat([(n1 - t1).reshape(-1), (n2 - t2).reshape(-1)])
        mx, e = float(err.abs().max()), _energy(h, n1, n2)
        if mx < tol:
            return n1, n2, e, mx
        vecs, errs = (vecs + [(n1, n2)])[-6:], (errs + [err])[-6:]
        m = len(vecs)
        if m == 1:
            t1, t2 = n1, n2
            continue
        B = np.zeros((m + 1, m + 1))
        for i in range(m):
            for j in range(i + 1):
                B[i, j] = B[j, i] = float(torch.vdot(errs[i], errs[j]).real)
        B[m, :m] = B[:m, m] = -1.0
        y = np.linalg.solve(B, np.append(np.zeros(m), -1.0))
        t1, t2 = (sum(float(y[k]) * vecs[k][q] for k in range(m)) for q in (0, 1))
    return t1, t2, e, mx


def _triples(h, t1, t2):
    """E(T) and each triple's energy at C(k,3) + C(j,2) + i"""
    o, v = t1.shape
    vvvo = h.block("vvvo").permute(3, 0, 1, 2).contiguous()  # [i, b, c, e]
    ovoo = h.block("ovoo").permute(2, 3, 0, 1).contiguous()  # [j, k, m, a]
    vvoo = h.block("vvoo").permute(2, 3, 0, 1).contiguous()  # [j, k, b, c]
    dv = h.ev[:, None, None] + h.ev[:, None] + h.ev
    out = torch.zeros(o * (o - 1) * (o - 2) // 6, dtype=torch.complex128, device=DEV)

    def pab(x):
        return x - x.transpose(0, 1) - x.transpose(0, 2)

    for k in range(2, o):
        for j in range(1, k):
            for i in range(j):
                c, d = 0, 0
                for p, q, r, s in ((i, j, k, 1), (j, i, k, -1), (k, j, i, -1)):
                    x = t2[q, r] @ vvvo[p].reshape(v * v, v).T - ovoo[q, r].T @ t2[p].reshape(o, v * v)
                    c = c + s * x.reshape(v, v, v)
                    d = d + s * t1[p][:, None, None] * vvoo[q, r]
                c, d = pab(c), pab(d)
                den = h.eo[i] + h.eo[j] + h.eo[k] - dv
                out[k * (k - 1) * (k - 2) // 6 + j * (j - 1) // 2 + i] = ((c + d).conj() * c / den).sum() / 6
    return complex(out.sum()), out


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "ccsd":
        if c["o"] + c["v"] > 200:  # above this the dense products take too long
            return None
        p = _problem(c["o"], c["v"], c["g"], seed)
        h = _Hamiltonian(p, c["real"])
        t = _amplitudes(p, seed)
        t1, t2, e, mx = _iterate(h, *(_real(*t) if c["real"] else t), c["iters"], c["shift"])
        return dict(t1=t1, t2=t2, energy=_number(e), max_dt=mx)
    if kind == "batch":
        got = []
        for k in range(c["n"]):
            h = _Hamiltonian(_problem(c["o"], c["v"], 1, seed, k), scale=0.5 + (k % 8) / 8.0)
            # the untrained model's guess is the first-order one
            got.append(_iterate(h, torch.zeros_like(h.D1, dtype=torch.complex128), h.block("vvoo").permute(2, 3, 0, 1) / h.D2,
                                c["iters"], 0.0))
        return dict(t1=torch.stack([g[0] for g in got]), t2=torch.stack([g[1] for g in got]), energy=np.array([_number(g[2]) for g in got]))
    if kind == "t3":
        if _t3_macs(c["o"], c["v"], 1) > 5e11:
            return None
        p = _problem(c["o"], c["v"], c["g"], seed)
        e, per = _triples(_Hamiltonian(p), *_amplitudes(p, seed))
        return dict(energy=_number(e), per_triple=per.cpu().numpy())
    if kind == "solve":
        h = _Hamiltonian(_problem(c["o"], c["v"], c["g"], seed, active=c["active"]), scale=0.4)
        _, _, e, _ = _iterate(h, torch.zeros_like(h.D1, dtype=torch.complex128), h.block("vvoo").permute(2, 3, 0, 1) / h.D2,
                              400, 2.0, 1e-10)
        return dict(energy=_number(e), heff=None, eig=None)  # the sector has its own dense oracle in the tests
    if kind == "zgemm":
        a, b = _zgemm_inputs(c, seed)
        return a @ b
    return None  # training visits the samples in an order of its own
