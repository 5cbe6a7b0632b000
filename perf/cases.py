"""What the matrix-element library is timed on: calls that its users' programs make.

A case is one call path of the public API (``paper_2106_12631_gb300.mg``) at one
process, precision and number of events:

* ``points``   |M|^2 of phase-space points that a generator hands over (``sigmakin``)
* ``bridge``   the same from an event record, with a helicity and a colour flow
               chosen per event (``matrix_elements_batch``)
* ``gradient`` d|M|^2 / d(uniforms) through autograd, forward and backward
* ``step``     one integration step on given uniforms: RAMBO, helicity filter,
               |M|^2, event sum, cross section
* ``generate`` unweighted events from device random numbers
* ``host``     the pipeline from host buffers to host results

Points of gg -> t t~ g (g), and the uniforms that a sampler proposes for them, pass
the usual generator cuts on the light partons (pT, rapidity, separation): without
them the matrix element diverges.

The mixed mode evaluates amplitudes in FP32, so a program that selects it keeps its
results as float32 (training targets, event weights); ``run`` stores them so.  The
FP64 mode's results stay float64.
"""
import math

import numpy as np
import torch

from paper_2106_12631_gb300 import mg

ECM = {"ee_mumu": 500.0, "gg_tt": 1500.0, "gg_ttg": 1500.0, "gg_ttgg": 1500.0}
NPAR = {"ee_mumu": 4, "gg_tt": 4, "gg_ttg": 5, "gg_ttgg": 6}
# floating-point operations of one event's |M|^2: colour-ordered off-shell currents
# summed before they are contracted, each once per helicity combination of its own
# legs; contractions per helicity; symmetric colour sum
FLOPS = {"ee_mumu": 1.5e3, "gg_tt": 5e3, "gg_ttg": 3.0e4, "gg_ttgg": 2.8e5}
RAMBO_FLOPS = 250.0  # per final particle


def listed():
    return [
        # the benchmark's batch of the heaviest process: one iteration of a production run
        dict(name="ttgg_mixed_large", kind="points", proc="gg_ttgg", mode="mixed", nevt=1 << 20),
        # an adaptive integrator's ordinary batch, of no round size
        dict(name="ttgg_mixed_ragged", kind="points", proc="gg_ttgg", mode="mixed", nevt=30011),
        # a sampler's single small request, where latency counts
        dict(name="ttgg_mixed_small", kind="points", proc="gg_ttgg", mode="mixed", nevt=64),
        # validation runs and programs that need full precision
        dict(name="ttgg_fp64", kind="points", proc="gg_ttgg", mode="fp64", nevt=32768),
        # event generator bridge: a record of events with helicity and colour-flow choices
        dict(name="ttgg_bridge_fp64", kind="bridge", proc="gg_ttgg", mode="fp64", nevt=4099),
        # the middle process in both precisions
        dict(name="ttg_mixed", kind="points", proc="gg_ttg", mode="mixed", nevt=262147),
        dict(name="ttg_fp64", kind="points", proc="gg_ttg", mode="fp64", nevt=50021),
        # training a sampler through the matrix element
        dict(name="ttg_gradient_mixed", kind="gradient", proc="gg_ttg", mode="mixed", nevt=1 << 17),
        # gradient checks and small fits in full precision
        dict(name="tt_gradient_fp64", kind="gradient", proc="gg_tt", mode="fp64", nevt=4097),
        # a total cross section on the device
        dict(name="tt_step_mixed", kind="step", proc="gg_tt", mode="mixed", nevt=1 << 20),
        # unweighted lepton events: tests' batch size, launches count
        dict(name="mumu_generate_fp64", kind="generate", proc="ee_mumu", mode="fp64", nevt=16384),
        # host programs that hold random numbers and results in their own memory
        dict(name="ttg_host_fp64", kind="host", proc="gg_ttg", mode="fp64", nevt=65536),
    ]


# per (kind, process, mode): the smallest and the largest number of events
RANGES = [
    ("points", "gg_ttgg", "mixed", 64, 1 << 20),
    ("points", "gg_ttgg", "fp64", 64, 32768),
    ("bridge", "gg_ttgg", "fp64", 64, 16384),
    ("points", "gg_ttg", "mixed", 64, 1 << 20),
    ("points", "gg_ttg", "fp64", 64, 1 << 17),
    ("bridge", "gg_ttg", "fp64", 64, 1 << 17),
    ("gradient", "gg_ttg", "mixed", 64, 1 << 17),
    ("gradient", "gg_ttg", "fp64", 64, 16384),
    ("gradient", "gg_tt", "mixed", 64, 1 << 17),
    ("gradient", "gg_tt", "fp64", 64, 32768),
    ("points", "gg_tt", "mixed", 64, 1 << 20),
    ("step", "gg_tt", "mixed", 64, 1 << 20),
    ("step", "gg_tt", "fp64", 64, 1 << 18),
    ("generate", "ee_mumu", "fp64", 64, 1 << 20),
    ("generate", "gg_tt", "fp64", 64, 1 << 18),
    ("host", "gg_tt", "fp64", 64, 1 << 18),
    ("host", "gg_ttg", "fp64", 64, 65536),
]


def draw(rng):
    kind, proc, mode, lo, hi = rng.choice(RANGES)
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.7:
        n = min(hi, n | 1)
    return dict(kind=kind, proc=proc, mode=mode, nevt=n)


def work(case):
    n, proc, kind = case["nevt"], case["proc"], case["kind"]
    npar, nf = NPAR[proc], NPAR[proc] - 2
    me, mom, rnd = 8 * n, 32 * npar * n, 32 * nf * n
    f = FLOPS[proc] * n
    if kind == "points":
        return {"bytes": mom + me, "flops": f}
    if kind == "bridge":
        return {"bytes": mom + me + (16 + 8) * n, "flops": f}
    if kind == "gradient":  # the forward pass's result, then the gradient (forward and adjoint)
        return {"bytes": 2 * rnd + 2 * me, "flops": 4 * f + 4 * RAMBO_FLOPS * nf * n}
    if kind == "step":
        return {"bytes": rnd + 2 * me, "flops": f + RAMBO_FLOPS * nf * n}
    if kind == "generate":
        return {"bytes": 2 * me, "flops": f + RAMBO_FLOPS * nf * n}
    return {"bytes": rnd + me, "flops": f + RAMBO_FLOPS * nf * n}


# ---- inputs -------------------------------------------------------------------------
def uniforms(seed, nrows, n, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return torch.rand((nrows, n), dtype=torch.float64, device=device, generator=g) * (1 - 2e-16) + 1e-16


def passes_cuts(mom):
    """Generator cuts on the final-state gluons (legs 4, ...): pT > 30 GeV, |y| < 4,
    separation > 0.4 from one another."""
    k = mom[4:]
    pt = torch.hypot(k[:, 1], k[:, 2])
    y = torch.asinh(k[:, 3] / pt)
    ok = ((pt > 30.0) & (y.abs() < 4.0)).all(0)
    for i in range(k.shape[0]):
        for j in range(i):
            dphi = torch.atan2(k[i, 2], k[i, 1]) - torch.atan2(k[j, 2], k[j, 1])
            dphi = torch.remainder(dphi + math.pi, 2 * math.pi) - math.pi
            ok &= torch.hypot(y[i] - y[j], dphi) > 0.4
    return ok


def fiducial(proc, n, seed):
    """Uniforms (nrows, n) whose phase-space points pass the cuts, and the momenta."""
    nrows = 4 * (NPAR[proc] - 2)
    rnds, moms, have, k = [], [], 0, 0
    while have < n:
        r = uniforms(seed * 1009 + k, nrows, min(max(4096, 2 * (n - have)), 1 << 19))
        m, _ = rambo64(r, proc)
        if NPAR[proc] > 4:
            ok = passes_cuts(m)
            r, m = r[:, ok], m[:, :, ok]
        r, m = r[:, : n - have], m[:, :, : n - have]
        rnds.append(r)
        moms.append(m)
        have += r.shape[1]
        k += 1
    return torch.cat(rnds, 1).contiguous(), torch.cat(moms, 2).contiguous()


def made(case, seed):
    """The case's inputs from its seed: what prepare hands over and exact starts from."""
    kind, proc, n = case["kind"], case["proc"], case["nevt"]
    if kind in ("points", "bridge", "gradient", "host"):
        rnd, mom = fiducial(proc, n, seed)
        return mom if kind in ("points", "bridge") else rnd
    return uniforms(seed, 4 * (NPAR[proc] - 2), n)


def good_helicities(proc):
    mom, _ = mg.rambo_seeded(proc, 16, ECM[proc], seed=7)
    return mg.filter_helicities(proc, mom)


def prepare(case, seed):
    kind, proc, n = case["kind"], case["proc"], case["nevt"]
    f64 = dict(dtype=torch.float64, device="cuda")
    s = dict(case=case, mask=good_helicities(proc), me=torch.empty(n, **f64))
    if kind == "points":
        s["mom"] = made(case, seed)
    elif kind == "bridge":
        s["record"] = made(case, seed).permute(2, 0, 1).contiguous()
        s["hel_rnd"], s["col_rnd"] = uniforms(seed + 1, 1, n)[0], uniforms(seed + 2, 1, n)[0]
        s["workspace"] = torch.empty(mg.batch_workspace_bytes(proc, n) // 8, **f64)
    elif kind == "gradient":
        s["rnd"] = made(case, seed).requires_grad_(True)
    elif kind == "generate":
        s["seed"] = seed
        s["mom"], s["wgt"] = torch.empty((NPAR[proc], 4, n), **f64), torch.empty(n, **f64)
    elif kind == "step":
        s["rnd"] = made(case, seed)
        s["mom"], s["wgt"] = torch.empty((NPAR[proc], 4, n), **f64), torch.empty(n, **f64)
    else:
        s["rnd"] = made(case, seed).cpu().pin_memory()
        nrows = 4 * (NPAR[proc] - 2)
        s["me"] = torch.empty(n, dtype=torch.float64, pin_memory=True)
        s["sums"] = torch.empty(3, dtype=torch.float64, pin_memory=True)
        s["workspace"] = torch.empty(mg.pipeline_workspace_bytes(proc, n, nrows) // 8, **f64)
    return s


def kept(case, x):
    """Results as the program keeps them: float32 from the mixed mode."""
    return x.to(torch.float32) if case["mode"] == "mixed" else x


def run(s):
    c = s["case"]
    proc, mode, ecm, kind = c["proc"], c["mode"], ECM[c["proc"]], c["kind"]
    if kind == "points":
        return kept(c, mg.sigmakin(proc, s["mom"], s["mask"], mode=mode, me=s["me"]))
    if kind == "bridge":
        me, hel, col = mg.matrix_elements_batch(proc, s["record"], s["mask"], mode=mode, hel_rnd=s["hel_rnd"],
                                                col_rnd=s["col_rnd"], me=s["me"], workspace=s["workspace"])
        return {"me": kept(c, me), "hel": hel, "col": col}
    if kind == "gradient":
        me = mg.matrix_element(s["rnd"], proc, ecm, s["mask"], mode)
        (grad,) = torch.autograd.grad(me.sum(), s["rnd"])
        return {"me": kept(c, me.detach()), "grad": kept(c, grad)}
    if kind == "step":
        mg.rambo(proc, s["rnd"], ecm, mom=s["mom"], wgt=s["wgt"])
        mask = mg.filter_helicities(proc, s["mom"][:, :, :16].contiguous())
        me = mg.sigmakin(proc, s["mom"], mask, mode=mode, me=s["me"])
        sums = mg.event_sum(me, s["wgt"])
        return {"me": kept(c, me), "wgt": s["wgt"], "xsec": kept(c, mg.cross_section(proc, ecm, sums))}
    if kind == "generate":
        mg.rambo_seeded(proc, c["nevt"], ecm, seed=s["seed"], mom=s["mom"], wgt=s["wgt"])
        me = mg.sigmakin(proc, s["mom"], s["mask"], mode=mode, me=s["me"])
        xsec = mg.cross_section(proc, ecm, mg.event_sum(me, s["wgt"]))
        idx, count = mg.unweight(me, s["wgt"], seed=s["seed"])
        events = torch.arange(c["nevt"], device=idx.device) < count  # entries of idx that are written
        return {"mom": s["mom"], "wgt": s["wgt"], "me": me, "xsec": xsec, "idx": torch.where(events, idx, -1),
                "count": count}
    mg.pipeline_host(proc, s["rnd"], ecm, s["mask"], mode=mode, me_host=s["me"], sums_host=s["sums"],
                     workspace=s["workspace"])
    torch.cuda.current_stream().synchronize()  # the program reads its host buffers next
    return {"me": s["me"], "sums": s["sums"]}


# ---- the same in 64 bits, in plain torch ---------------------------------------------
MZ, WZ, ALPHA_INV, SW2, MT, WT, ALPHA_S = 91.188, 2.441, 132.507, 0.2222, 173.0, 1.491, 0.118
E2 = 4 * math.pi / ALPHA_INV
GS = math.sqrt(4 * math.pi * ALPHA_S)


def rambo64(r, proc):
    """Momenta (npar, 4, n) and flat phase-space weights of uniforms (4 nf, n)."""
    ecm, nf = ECM[proc], NPAR[proc] - 2
    ms = [MT, MT] + [0.0] * (nf - 2) if proc != "ee_mumu" else [0.0, 0.0]
    c = 2 * r[0::4] - 1
    st, phi, e = torch.sqrt(1 - c * c), 2 * math.pi * r[1::4], -torch.log(r[2::4] * r[3::4])
    q = torch.stack([e, e * st * torch.cos(phi), e * st * torch.sin(phi), e * c], 1)
    Q = q.sum(0)
    M = torch.sqrt(Q[0] ** 2 - Q[1] ** 2 - Q[2] ** 2 - Q[3] ** 2)
    b, g, x = -Q[1:] / M, Q[0] / M, ecm / M
    bq = (b * q[:, 1:]).sum(1)
    p0 = x * (g * q[:, 0] + bq)
    pv = x * (q[:, 1:] + b * q[:, 0:1] + (bq / (1 + g)).unsqueeze(1) * b)
    w = (math.pi / 2) ** (nf - 1) * ecm ** (2 * nf - 4) / (math.factorial(nf - 1) * math.factorial(nf - 2))
    w = torch.full_like(p0[0], w)
    if any(ms):
        m2 = torch.tensor(ms, dtype=r.dtype, device=r.device).unsqueeze(1) ** 2
        pd = p0.detach()
        xi = torch.full_like(pd[0], math.sqrt(1 - (sum(ms) / ecm) ** 2))
        for _ in range(12):
            en = torch.sqrt(m2 + (xi * pd) ** 2)
            xi = xi - (en.sum(0) - ecm) / (xi * pd ** 2 / en).sum(0)
        # one more step on the graph: the implicit function's derivative
        en = torch.sqrt(m2 + (xi * p0) ** 2)
        xi = xi - (en.sum(0) - ecm) / (xi * pd ** 2 / torch.sqrt(m2 + (xi * pd) ** 2)).sum(0)
        kk = xi * p0
        k0, kv = torch.sqrt(m2 + kk ** 2), xi * pv
        w = w * xi ** (2 * nf - 3) * (kk / k0).prod(0) / (kk ** 2 / k0).sum(0) * ecm
    else:
        k0, kv = p0, pv
    h, z = torch.full_like(k0[0], ecm / 2), torch.zeros_like(k0[0])
    beams = torch.stack([torch.stack([h, z, z, h]), torch.stack([h, z, z, -h])])
    return torch.cat([beams, torch.cat([k0.unsqueeze(1), kv], 1)], 0), w


def chain_colours(ng):
    """Colour matrix of the ng! chains (T^{a_s1} .. T^{a_sng})_ij in lexicographic order."""
    import itertools
    lam = np.zeros((8, 3, 3), complex)
    for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        a = (0, 3, 5)[k]
        lam[a, i, j] = lam[a, j, i] = 1
        lam[a + 1, i, j], lam[a + 1, j, i] = -1j, 1j
    # the two diagonal generators, in the positions left over
    free = [a for a in range(8) if not lam[a].any()]
    lam[free[0]], lam[free[1]] = np.diag([1, -1, 0]), np.diag([1, 1, -2]) / math.sqrt(3)
    T = lam / 2
    perms = list(itertools.permutations(range(ng)))
    chains = []
    for p in perms:
        t = np.eye(3, dtype=complex)[None]
        for _ in p:
            t = np.einsum("aij,bjk->abik", t, T).reshape(-1, 3, 3)
        t = t.reshape((8,) * ng + (9,))
        chains.append(np.transpose(t, [p.index(k) for k in range(ng)] + [ng]).reshape(-1))
    ch = np.array(chains)
    return perms, (ch @ ch.conj().T).real


def mdot(a, b):
    return a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3]


class Ordered64:
    """Colour-ordered amplitudes of top, antitop and gluons from off-shell currents in
    Feynman gauge.  Every current has one axis of length 2 (or 1) per leg for that leg's
    spin state and the events last; spin states need not be helicities for the sum."""

    def __init__(self, mom):
        self.n = mom.shape[0]
        self.mom = mom
        self.gl = [l for l in range(self.n) if l not in (2, 3)]
        self.sign = [-1 if l < 2 else 1 for l in range(self.n)]
        self.memo = {}

    def lift(self, leg, states):
        """Two states of four components (tensors over events) -> one current."""
        shape = [1] * self.n + [-1]
        shape[leg] = 2
        return tuple(torch.stack([s[k] for s in states]).reshape(shape) for k in range(4))

    def K(self, legs):
        return sum(self.sign[l] * self.mom[l] for l in legs)

    def gluon(self, w):
        if ("g", w) in self.memo:
            return self.memo["g", w]
        if len(w) == 1:
            k = self.mom[w[0]]
            kt = torch.sqrt(k[1] ** 2 + k[2] ** 2)
            kk = torch.sqrt(kt ** 2 + k[3] ** 2)
            on = kt > 0
            one = torch.ones_like(kt)
            safe = torch.where(on, kt, one)
            cp, sp = torch.where(on, k[1] / safe, one), torch.where(on, k[2] / safe, 0 * one)
            ct, sth = k[3] / kk, torch.where(on, kt / kk, 0 * one)
            z = torch.zeros_like(kt)
            states = [(z, ct * cp, ct * sp, -sth), (z, -sp, cp, z)]
            out = self.lift(w[0], [tuple(x + 0j for x in s) for s in states])
        else:
            acc = [0, 0, 0, 0]
            for i in range(1, len(w)):
                a, b = self.gluon(w[:i]), self.gluon(w[i:])
                ka, kb = self.K(w[:i]), self.K(w[i:])
                ab, c1, c2 = mdot(a, b), mdot(ka + 2 * kb, a), mdot(2 * ka + kb, b)
                for m in range(4):
                    acc[m] = acc[m] - 1j * GS * (ab * (kb[m] - ka[m]) - c1 * b[m] + c2 * a[m])
                for j in range(i + 1, len(w)):
                    b, c = self.gluon(w[i:j]), self.gluon(w[j:])
                    ab, ac, bc = mdot(a, b), mdot(a, c), mdot(b, c)
                    for m in range(4):
                        acc[m] = acc[m] - 1j * GS * GS * (bc * a[m] + ab * c[m] - 2 * ac * b[m])
            k = self.K(w)
            pr = -1j / mdot(k, k)
            out = tuple(x * pr for x in acc)
        self.memo["g", w] = out
        return out

    def spinors(self, leg, anti):
        p = self.mom[leg]
        root = torch.sqrt(2 * (p[0] + MT))
        z = torch.zeros_like(p[0]) + 0j
        states = []
        for s in (0, 1):
            # (p.sigma + m) chi / sqrt(2 (E + m)) and the same with sigma-bar
            lo = [(p[0] - p[3] + MT) + z, -(p[1] + 1j * p[2])] if s == 0 else [-(p[1] - 1j * p[2]), p[0] + p[3] + MT + z]
            hi = [(p[0] + p[3] + MT) + z, p[1] + 1j * p[2]] if s == 0 else [p[1] - 1j * p[2], p[0] - p[3] + MT + z]
            lo, hi = [x / root for x in lo], [x / root for x in hi]
            states.append((lo[0], lo[1], -hi[0], -hi[1]) if anti
                          else (hi[0].conj(), hi[1].conj(), lo[0].conj(), lo[1].conj()))
        return self.lift(leg, states)

    @staticmethod
    def row_slash(f, V):
        vp, vm = V[0] + V[3], V[0] - V[3]
        pl, mi = V[1] + 1j * V[2], V[1] - 1j * V[2]
        return (f[2] * vp + f[3] * pl, f[2] * mi + f[3] * vm, f[0] * vm - f[1] * pl, f[1] * vp - f[0] * mi)

    def row(self, w):
        """Off-shell top line with gluons w attached, in this order from the top."""
        if ("r", w) in self.memo:
            return self.memo["r", w]
        if not w:
            out = self.spinors(2, False)
        else:
            acc = self.joined(w)
            k = self.K((2,) + w)
            kk = [x + 0j for x in k]
            s = self.row_slash(acc, kk)
            pr = 1j / (mdot(k, k) - MT * MT + 1j * MT * WT)
            out = tuple((s[m] + MT * acc[m]) * pr for m in range(4))
        self.memo["r", w] = out
        return out

    def joined(self, w):
        acc = [0, 0, 0, 0]
        for j in range(len(w)):
            s = self.row_slash(self.row(w[:j]), self.gluon(w[j:]))
            acc = [acc[m] + 1j * GS * s[m] for m in range(4)]
        return acc

    def squared(self):
        """|M|^2 summed over spins and colours."""
        perms, C = chain_colours(len(self.gl))
        v = self.spinors(3, True)
        J = []
        for p in perms:
            f = self.joined(tuple(self.gl[k] for k in p))
            J.append(f[0] * v[0] + f[1] * v[1] + f[2] * v[2] + f[3] * v[3])
        J = torch.stack([x.expand([2] * self.n + [-1]) for x in J])
        shape = J.shape
        J = torch.view_as_real(J.reshape(shape[0], -1)).reshape(shape[0], -1)
        Cd = torch.tensor(C, dtype=torch.float64, device=J.device)
        t = (J * (Cd @ J)).reshape(-1, shape[-1], 2)
        return t.sum((0, 2))


def me64(mom, proc):
    if proc == "ee_mumu":
        s = mdot(mom[0] + mom[1], mom[0] + mom[1])
        t, u = -2 * mdot(mom[1], mom[3]), -2 * mdot(mom[1], mom[2])
        gz2, gl, gr = E2 / (SW2 * (1 - SW2)), -0.5 + SW2, SW2
        D = s - MZ * MZ + 1j * MZ * WZ
        tot = 0
        for a in (gl, gr):
            for b in (gl, gr):
                tot = tot + 4 * (u if a == b else t) ** 2 * (E2 / s + gz2 * a * b / D).abs() ** 2
        return tot / 4
    sym = 2 if proc == "gg_ttgg" else 1
    return Ordered64(mom).squared() / (4 * 64 * sym)


def exact(case, seed):
    kind, proc, n = case["kind"], case["proc"], case["nevt"]
    ecm, nf = ECM[proc], NPAR[proc] - 2
    if kind == "generate":
        # the device's counter-based uniforms, from the generator's published definition
        rnd = torch.from_numpy(counter_uniforms(seed, 4 * nf, n)).cuda()
    else:
        x = made(case, seed)
        rnd = x if kind not in ("points", "bridge") else None
    step = 1 << (13 if proc == "gg_ttgg" else 14)
    me, wgt, moms, grad = [], [], [], []
    for i in range(0, n, step):
        if rnd is None:
            me.append(me64(x[:, :, i:i + step], proc))
            continue
        r = rnd[:, i:i + step].clone().requires_grad_(kind == "gradient")
        mom, w = rambo64(r, proc)
        m = me64(mom, proc)
        if kind == "gradient":
            grad.append(torch.autograd.grad(m.sum(), r)[0])
        me.append(m.detach())
        wgt.append(w.detach())
        moms.append(mom.detach())
    me = torch.cat(me)
    if kind == "points":
        return me
    if kind == "bridge":
        return {"me": me, "hel": None, "col": None}
    if kind == "gradient":
        return {"me": me, "grad": torch.cat(grad, 1)}
    wgt = torch.cat(wgt)
    x = wgt * me
    sums = torch.stack([x.sum(), (x * x).sum(), torch.full_like(x[0], float(n))])
    if kind == "host":
        return {"me": me, "sums": sums}
    norm = 0.3893793721e9 * (2 * math.pi) ** (4 - 3 * nf) / (2 * ecm * ecm)
    err = torch.sqrt(((x - x.mean()) ** 2).sum() / (n - 1) / n) if n > 1 else torch.zeros_like(x[0])
    xsec = torch.stack([norm * x.mean(), norm * err])
    if kind == "step":
        return {"me": me, "wgt": wgt, "xsec": xsec}
    return {"mom": torch.cat(moms, 2), "wgt": wgt, "me": me, "xsec": xsec, "idx": None, "count": None}


def counter_uniforms(seed, nrows, n):
    """SplitMix64 as a counter-based generator: event i, row k uses counter 64 i + k + 1."""
    def mix(z):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))
    with np.errstate(over="ignore"):
        key = mix(np.array([seed], dtype=np.uint64))[0]
        ev = np.arange(n, dtype=np.uint64) * np.uint64(64)
        rows = [mix(key + (ev + np.uint64(k + 1)) * np.uint64(0x9E3779B97F4A7C15)) for k in range(nrows)]
    return np.stack([((z >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for z in rows])
