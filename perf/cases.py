"""The work that users of this library have it do, as measurable cases.

Every case goes through the package's public calls on seeded inputs of the
shapes that the library's workloads, tests and benchmark use: one frozen
natural orbital step is D_vv and E_vv (dsrg_fno_vv_opdm), the natural orbitals
and their cut (dsrg_fno_truncate), and the correction for the discarded
orbitals (dsrg_fno_discarded_correction).  Beside them stand the energy by
itself, the ladder in the kept orbitals, the compressed auxiliary basis and the
batch of ragged instances.  The fast form is what production runs use; the
float64 form is the one results are checked with.

Inputs follow the recipe of synth/problems.py (decaying normal DF factors,
uniform orbital energies per block), drawn on the device.  The state-averaged
densities are those of an ensemble of closed-shell determinants in random
active orbital bases, so Gamma1 and the 2-cumulant are exact and dense.

An orbital is fixed only as well as its occupation number is separated from
the next.  Where the density matrix is an input, the natural orbitals are
returned multiplied by their occupation numbers, the weight they enter later
steps with.  In a whole step they are an intermediate between two roundings
(of D_vv and of its eigenvectors), and what is fixed by the inputs is returned:
the density, the occupation numbers, and the energies in the kept orbitals.
"""
import math
import random

import numpy as np
import torch

import paper_2312_07008_gb300 as pkg

S_FLOW = 0.5        # flow parameter of every workload here
DEGEN = 0.01        # near-degeneracy ratio of the cut


def listed():
    return [
        # the smallest whole step: a small closed-shell molecule, where launches and waits count
        dict(name="step_sr_nocc10_nvir90", kind="step", ncore=10, nact=0, nvir=90, naux=300, states=1, po=98.5, fast=True),
        # a whole step of an ordinary state-averaged molecule
        dict(name="step_cas6_nvir300", kind="step", ncore=20, nact=6, nvir=300, naux=1000, states=3, po=98.5, fast=True),
        # the same density in the plain float64 form, the one that results are checked with
        dict(name="opdm_fp64_cas6_nvir300", kind="opdm", ncore=20, nact=6, nvir=300, naux=1000, states=3, fast=False),
        # the density of a large molecule in a large basis: what most of the time goes into
        dict(name="opdm_cas10_nvir1200", kind="opdm", ncore=60, nact=10, nvir=1200, naux=3600, states=4, fast=True),
        # the energy alone, as at further geometries; odd sizes
        dict(name="energy_cas5_nvir443", kind="energy", ncore=37, nact=5, nvir=443, naux=1455, states=2, fast=True),
        # natural orbitals of a large basis and of a kept basis
        dict(name="truncate_1200", kind="truncate", nvir=1200, po=98.0),
        dict(name="truncate_203", kind="truncate", nvir=203, po=99.0),
        # the discarded-orbital correction of the large molecule at its 99 % cut
        dict(name="correction_cas10_nvir1200_kept203", kind="correction", ncore=60, nact=10, nvir=1200, naux=3600, states=4,
             nkept=203, fast=True),
        # the four-virtual term of the next step in a kept basis of odd size
        dict(name="ladder_nv119", kind="ladder", nv=119, naux=1500, npairs=820),
        # natural auxiliary functions of the ordinary molecule
        dict(name="naf_naux400", kind="naf", nh=26, np=306, naux=400, keep=0.75),
        # a scan over many molecules of different sizes, each a whole step
        dict(name="batch_ragged8", kind="batch", count=8, sizes_seed=38, po=98.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "opdm", "energy", "truncate", "correction", "ladder", "naf", "batch"])
    if kind in ("step", "opdm", "energy", "correction"):
        while True:
            c = dict(kind=kind, ncore=_log_int(rng, 6, 95), nact=rng.choice([0, 4, 5, 6, 8, 10]), nvir=_log_int(rng, 70, 1200),
                     states=rng.randint(2, 5), fast=True)
            c["naux"] = rng.randint(2 * (c["ncore"] + c["nact"] + c["nvir"]), 4 * (c["ncore"] + c["nact"] + c["nvir"]))
            if work(dict(c, kind="opdm"))["flops"] <= 4e12:
                break
        if kind == "step":
            c["po"] = rng.choice([98.0, 98.5, 99.0])
        if kind == "correction":
            c["nkept"] = max(1, int(c["nvir"] * rng.uniform(0.15, 0.6)))
        if kind == "opdm" and work(c)["flops"] < 2e11:
            c["fast"] = rng.random() < 0.5
        return c
    if kind == "truncate":
        return dict(kind=kind, nvir=_log_int(rng, 60, 1200), po=rng.choice([98.0, 98.5, 99.0]))
    if kind == "ladder":
        return dict(kind=kind, nv=_log_int(rng, 30, 150), naux=rng.randint(300, 2000), npairs=rng.randint(50, 1200))
    if kind == "naf":
        nh, np_ = rng.randint(16, 40), rng.randint(100, 400)
        return dict(kind=kind, nh=nh, np=np_, naux=_log_int(rng, 150, 400), keep=rng.choice([0.5, 0.75, 0.9]))
    while True:
        c = dict(kind="batch", count=rng.randint(4, 8), sizes_seed=rng.randint(0, 10 ** 6), po=98.5)
        if work(c)["flops"] <= 1e13:
            return c


# ------------------------------------------------------------------ inputs
def _densities(nact, states, g):
    """Gamma1 and Lambda2 of an equally weighted ensemble of closed-shell
    determinants, each in its own random orbital basis."""
    nocc = nact // 2
    g1 = np.zeros((nact, nact))
    g2 = np.zeros((nact,) * 4)
    for _ in range(states):
        q, _ = np.linalg.qr(g.standard_normal((nact, nact)))
        p = 2.0 * q[:, :nocc] @ q[:, :nocc].T
        g1 += p / states
        g2 += (np.einsum("pr,qs->pqrs", p, p) - 0.5 * np.einsum("ps,qr->pqrs", p, p)) / states
    l2 = g2 - np.einsum("pr,qs->pqrs", g1, g1) + 0.5 * np.einsum("ps,qr->pqrs", g1, g1)
    return g1, l2


def _molecule(c, seed):
    """Device tensors of one problem: B, eps, gamma1, lambda2."""
    nc, na, nv, nq = c["ncore"], c["nact"], c["nvir"], c["naux"]
    g = np.random.default_rng(seed)
    eps = np.concatenate([np.sort(g.uniform(-2.0, -0.3, nc)), np.sort(g.uniform(-0.5, 0.3, na)), np.sort(g.uniform(0.1, 5.0, nv))])
    g1, l2 = _densities(na, c["states"], g) if na else (None, None)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B = torch.randn((nq, nc + na, na + nv), dtype=torch.float64, device="cuda", generator=gen)
    if na:
        z = B[:, nc:, :na].clone()
        B[:, nc:, :na] = (z + z.transpose(1, 2)) / math.sqrt(2.0)
    loc = lambda a, b: torch.cat([torch.arange(a, device="cuda"), torch.arange(b, device="cuda")]).double()  # noqa: E731
    B *= 0.05 * torch.exp(-0.01 * (loc(nc, na)[:, None] + loc(na, nv)[None, :]))
    up = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return B, up(eps), up(g1), up(l2)


def _problem(c, t):
    form = pkg.SLICED_BF16 if c.get("fast", True) else pkg.FP64
    return pkg.Problem(c["ncore"], c["nact"], c["nvir"], c["naux"], t[0], t[1], t[2], t[3],
                       weights=np.full(c["states"], 1.0 / c["states"]), s=S_FLOW, precision=form)


def _density_matrix(n, seed):
    """A matrix like D_vv: a sum of squares whose rows decay with the orbital energy."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((n, 4 * n), dtype=torch.float64, device="cuda", generator=gen)
    z *= 0.7 * torch.exp(-0.01 * torch.arange(n, device="cuda").double())[:, None] / math.sqrt(n)
    d = z @ z.T
    return 0.5 * (d + d.T)


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


def _batch_members(c):
    rng = random.Random(c["sizes_seed"])
    out = []
    for _ in range(c["count"]):
        m = dict(ncore=rng.randint(10, 60), nact=rng.choice([0, 4, 6, 8]), nvir=rng.randint(100, 800), states=rng.randint(2, 5))
        m["naux"] = 3 * (m["ncore"] + m["nact"] + m["nvir"])
        out.append(m)
    return out


def prepare(case, seed):
    c, k = case, case["kind"]
    st = dict(case=case)
    if k in ("step", "opdm", "energy", "correction"):
        t = _molecule(c, seed)
        st["prob"] = _problem(c, t)
        nv = c["nvir"]
        if k in ("step", "opdm"):
            st["d"] = _empty(nv, nv)
        if k == "step":
            st["on"], st["no"] = _empty(nv), _empty(nv, nv)
        if k == "correction":
            # the NOs that the program has from its truncation, and its E_vv
            w, v = torch.linalg.eigh(_density_matrix(nv, seed + 1))
            st["no"] = v.flip(1).contiguous()
            st["e2"] = -80000.0
            st["eps_out"] = _empty(c["nkept"])
    elif k == "truncate":
        n = c["nvir"]
        st.update(d=_density_matrix(n, seed), on=_empty(n), no=_empty(n, n))
    elif k == "ladder":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        b = 0.05 * torch.randn((c["naux"], c["nv"], c["nv"]), dtype=torch.float64, device="cuda", generator=gen)
        st["B"] = (0.5 * (b + b.transpose(1, 2))).contiguous()
        st["T"] = 0.05 * torch.randn((c["npairs"], c["nv"], c["nv"]), dtype=torch.float64, device="cuda", generator=gen)
        st["C"] = torch.empty_like(st["T"])
    elif k == "naf":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        b = torch.randn((c["naux"], c["nh"], c["np"]), dtype=torch.float64, device="cuda", generator=gen)
        b *= 0.05 * torch.exp(-0.01 * (torch.arange(c["nh"], device="cuda").double()[:, None]
                                       + torch.arange(c["np"], device="cuda").double()[None, :]))
        # functions of decreasing weight, as an auxiliary basis has them
        b *= torch.exp(-1.5 * torch.arange(c["naux"], device="cuda").double() / c["naux"])[:, None, None]
        w = torch.sort((b * b).sum((1, 2)), descending=True).values
        st.update(B=b, out=torch.zeros_like(b), w=_empty(c["naux"]), thr=float(w[int(c["keep"] * c["naux"]) - 1]))
    else:
        ms = _batch_members(c)
        ts = [_molecule(m, seed * 100 + i) for i, m in enumerate(ms)]
        st["probs"] = [_problem(m, t) for m, t in zip(ms, ts)]
        st["d"] = [_empty(m["nvir"], m["nvir"]) for m in ms]
        st["on"] = [_empty(m["nvir"]) for m in ms]
        st["no"] = [_empty(m["nvir"], m["nvir"]) for m in ms]
    return st


def run(state):
    c, k = state["case"], state["case"]["kind"]
    if k == "step":
        p, d, on, no = state["prob"], state["d"], state["on"], state["no"]
        e2 = pkg.dsrg_fno_vv_opdm(p, d)
        n = pkg.dsrg_fno_truncate(c["nvir"], d, pkg.MODE_PO, c["po"], DEGEN, on, no)
        de, ef = pkg.dsrg_fno_discarded_correction(p, n, no, e2_mo=e2)
        return dict(e2=e2, d=d, on=on, nkept=n, de=de, e2_fno=ef)
    if k == "opdm":
        return dict(e2=pkg.dsrg_fno_vv_opdm(state["prob"], state["d"]), d=state["d"])
    if k == "energy":
        return dict(e2=pkg.dsrg_fno_pt2_energy(state["prob"]))
    if k == "truncate":
        n = pkg.dsrg_fno_truncate(c["nvir"], state["d"], pkg.MODE_PO, c["po"], DEGEN, state["on"], state["no"])
        return dict(on=state["on"], no=state["no"] * state["on"], nkept=n)
    if k == "correction":
        de, ef = pkg.dsrg_fno_discarded_correction(state["prob"], c["nkept"], state["no"], e2_mo=state["e2"],
                                                   eps_fno_out=state["eps_out"])
        return dict(de=de, e2_fno=ef, eps=state["eps_out"])
    if k == "ladder":
        pkg.dsrg_fno_ladder(state["B"], state["T"], state["C"])
        return dict(c=state["C"])
    if k == "naf":
        n = pkg.dsrg_fno_naf(c["nh"], c["np"], c["naux"], state["B"], state["thr"], pkg.SLICED_BF16, state["out"], state["w"])
        return dict(naux=n, w=state["w"], b=state["out"])
    r = pkg.dsrg_fno_batch_run(state["probs"], state["d"], (pkg.MODE_PO, c["po"], DEGEN), state["on"], state["no"], True)
    return dict(e2=[x["e2"] for x in r], nkept=[x["nkept"] for x in r], de=[x["de"] for x in r], d=state["d"], on=state["on"])


# ------------------------------------------------------------------ work
def _sum_work(parts):
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


def work(case):
    """Inputs read and outputs written once; multiplications and additions of
    the equations: every unordered hole pair's integrals, the update of D_vv
    (symmetric), a tridiagonal reduction with back-transformation (4 n^3 + ...)
    for an eigensolve, the rotation of B and the energy in the kept basis."""
    c, k = case, case["kind"]
    if k in ("step", "opdm", "energy", "correction"):
        nh, np_, nv, nq = c["ncore"] + c["nact"], c["nact"] + c["nvir"], c["nvir"], c["naux"]
        pairs = nh * (nh + 1) // 2
        b_in = 8.0 * nq * nh * np_
        integrals = 2.0 * nq * pairs * np_ * np_
        energy_f = lambda n: 2.0 * nq * pairs * n * n  # noqa: E731
        opdm = dict(bytes=b_in + 8.0 * nv * nv, flops=integrals + 1.0 * nh * nh * nv ** 3)
        corr = lambda n: dict(bytes=b_in + 8.0 * nv * n, flops=2.0 * nq * nh * nv * n + energy_f(n) + 4.0 * n ** 3)  # noqa: E731
        if k == "opdm":
            return opdm
        if k == "energy":
            return dict(bytes=b_in, flops=energy_f(nv))
        if k == "correction":
            return corr(c["nkept"])
        return _sum_work([opdm, work(dict(kind="truncate", nvir=nv)), corr(nv // 2)])
    if k == "truncate":
        return dict(bytes=24.0 * c["nvir"] ** 2, flops=4.0 * c["nvir"] ** 3)
    if k == "ladder":
        nv = c["nv"]
        return dict(bytes=8.0 * nv * nv * (c["naux"] + 2 * c["npairs"]), flops=2.0 * nv ** 4 * (c["naux"] + c["npairs"]))
    if k == "naf":
        nq, L = c["naux"], c["nh"] * c["np"]
        return dict(bytes=8.0 * nq * L * (1 + c["keep"]), flops=nq * nq * L + 2.0 * c["keep"] * nq * nq * L + 4.0 * nq ** 3)
    return _sum_work([work(dict(m, kind="step")) for m in _batch_members(c)])


# ------------------------------------------------------------------ 64 bits
def _reg(delta):
    x = S_FLOW * delta * delta
    big = torch.where(delta == 0, torch.ones_like(delta), delta)
    return torch.where(x < 1e-3, S_FLOW * delta * (1 - x * (0.5 - x * (1 / 6 - x * (1 / 24 - x / 120)))), -torch.expm1(-x) / big)


def _amplitudes(B, eps, nc, na, want_ts):
    """tau and kappa [i][j][a][b] over virtuals, and t^{ij}_{ex} (e virtual, x active)."""
    nq, nh, np_ = B.shape
    nv = np_ - na
    Bv = B[:, :, na:].contiguous()
    ea, ev = eps[nc:nc + na], eps[nh:]
    tau, kap = B.new_empty((nh, nh, nv, nv)), B.new_empty((nh, nh, nv, nv))
    ts = B.new_empty((nh, nh, nv, na)) if want_ts and na else None
    for i in range(nh):
        left = Bv[:, i, :].T
        nu = (left @ Bv.reshape(nq, nh * nv)).reshape(nv, nh, nv).transpose(0, 1)
        dl = eps[i] + eps[:nh][:, None, None] - ev[None, :, None] - ev[None, None, :]
        tau[i] = nu * _reg(dl)
        kap[i] = 2 * nu - dl * tau[i]
        if ts is not None:
            nu = (left @ B[:, :, :na].reshape(nq, nh * na)).reshape(nv, nh, na).transpose(0, 1)
            ts[i] = nu * _reg(eps[i] + eps[:nh][:, None, None] - ev[None, :, None] - ea[None, None, :])
    return tau, kap, ts


def _holes(c, g1, l2, dev):
    gam = 2.0 * torch.eye(c["ncore"] + c["nact"], dtype=torch.float64, device=dev)
    if c["nact"]:
        gam[c["ncore"]:, c["ncore"]:] = g1
    return gam


def _dress(tau, gam, l2, nc, na):
    """W^{ij} = sum_kl Gamma^{kl}_{ij} tau^{kl} with the hole 2-RDM."""
    nh, nv = tau.shape[0], tau.shape[2]
    w = tau.clone()
    w[:nc] *= 2.0
    w[:, :nc] *= 2.0
    if na:
        g = gam[nc:, nc:]
        w[nc:] = torch.einsum("ki,kjab->ijab", g, w[nc:])
        w[:, nc:] = torch.einsum("lj,ilab->ijab", g, w[:, nc:])
    out = w - 0.5 * w.transpose(0, 1)
    if na:
        out[nc:, nc:] += torch.einsum("klij,klab->ijab", l2, tau[nc:, nc:])
    return out


def _exact_energy(B, eps, gam, l2, nc, na):
    tau, kap, _ = _amplitudes(B, eps, nc, na, False)
    return 0.5 * float((_dress(tau, gam, l2, nc, na) * kap).sum())


def _exact_opdm(c, B, eps, g1, l2):
    nc, na, nv = c["ncore"], c["nact"], c["nvir"]
    nh = nc + na
    gam = _holes(c, g1, l2, B.device)
    tau, kap, ts = _amplitudes(B, eps, nc, na, True)
    w = _dress(tau, gam, l2, nc, na)
    e2 = 0.5 * float((w * kap).sum())
    del kap
    d = B.new_zeros((nv, nv))
    for i in range(nh):
        d += torch.einsum("jag,jbg->ab", w[i], tau[i])
    del tau, w
    if na:
        G, L, Th = g1, l2, 2.0 * torch.eye(na, dtype=torch.float64, device=B.device) - g1
        tc = 2.0 * ts - ts.transpose(0, 1)
        es = torch.einsum
        f = eps[nc:nh][None, :] - eps[nc:nh][:, None]     # [u][x] eps_x - eps_u
        t1 = 0.5 * es("ux,xu,iuex->ie", f, G, tc[:, nc:]) * _reg(eps[:nh][:, None] - eps[nh:][None, :])
        tm, tu = t1[:nc], t1[nc:]
        aa, mm = ts[nc:, nc:], ts[:nc, :nc]
        ma, am = ts[:nc, nc:], ts[nc:, :nc].transpose(0, 1)   # [m][u]: t^{mu}, t^{um}
        d += 2.0 * tm.T @ tm + tu.T @ G @ tu
        d += es("ue,uvxy,xyfv->ef", tu, L, aa) + es("uvey,uvxy,xf->ef", aa, L, tu)
        d += es("mnev,uv,mnfu->ef", mm, Th, tc[:nc, :nc])
        p, q = es("muey,uv,xy->mvex", ma, G, Th), es("muey,uv,xy->mvex", am, G, Th)
        d += 0.5 * es("mvex,mvfx->ef", p, 2 * ma - am) + 0.5 * es("mvex,mvfx->ef", q, 2 * am - ma)
        d += es("mvey,uvxy,mxfu->ef", ma, L, 2 * ma - am) - es("mvey,uvxy,mxfu->ef", am, L, ma)
        d -= es("mvex,uvxy,myfu->ef", am, L, am)
        z = es("uvez,wz->uvew", aa, Th)
        ta = 2.0 * aa - aa.transpose(0, 1)
        d += 0.5 * es("uvew,uvxy,xyfw->ef", z, L, aa) + 0.25 * es("uxew,uv,xy,vyfw->ef", z, G, G, ta)
        ga = es("wvey,wz->zvey", aa, G)      # first hole dressed
        gb = es("vwey,wz->vzey", aa, G)      # second hole dressed
        d += 0.5 * es("zvey,uvxy,zxfu->ef", ga, L, ta) - 0.5 * es("vzey,uvxy,zxfu->ef", gb, L, aa)
        d -= 0.5 * es("vzex,uvxy,yzfu->ef", gb, L, aa)
    return e2, 0.5 * (d + d.T)


def _exact_truncate(d, po):
    w, v = torch.linalg.eigh(d)
    w, v = w.flip(0), v.flip(1)
    top = v.gather(0, v.abs().argmax(0, keepdim=True))
    v = v * torch.where(top < 0, -1.0, 1.0)
    on = w.cpu().numpy()
    n = min(len(on), int(np.searchsorted(np.cumsum(on), po / 100.0 * on.sum())) + 1)
    while 0 < n < len(on) and on[n - 1] - on[n] < DEGEN * max(on[n - 1], on[n]):
        n += 1
    return w, v, n


def _exact_correction(c, B, eps, g1, l2, no, n):
    nc, na = c["ncore"], c["nact"]
    nh = nc + na
    vk = no[:, :n]
    e, w = torch.linalg.eigh(vk.T @ (eps[nh:, None] * vk))
    bf = torch.cat([B[:, :, :na], B[:, :, na:] @ (vk @ w)], 2)
    return _exact_energy(bf, torch.cat([eps[:nh], e]), _holes(c, g1, l2, B.device), l2, nc, na), e


def _exact_step(c, t, po):
    e2, d = _exact_opdm(c, *t)
    on, no, n = _exact_truncate(d, po)
    ef, _ = _exact_correction(c, *t, no, n)
    return dict(e2=e2, d=d, on=on, nkept=None, de=e2 - ef, e2_fno=ef)


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("step", "opdm", "energy") and work(c)["flops"] > 2e12:
        return None
    if k in ("step", "opdm", "energy", "correction"):
        t = _molecule(c, seed)
        if k == "step":
            return _exact_step(c, t, c["po"])
        if k == "opdm":
            e2, d = _exact_opdm(c, *t)
            return dict(e2=e2, d=d)
        if k == "energy":
            return dict(e2=_exact_energy(t[0], t[1], _holes(c, t[2], t[3], "cuda"), t[3], c["ncore"], c["nact"]))
        _, v = torch.linalg.eigh(_density_matrix(c["nvir"], seed + 1))
        ef, e = _exact_correction(c, *t, v.flip(1).contiguous(), c["nkept"])
        return dict(de=-80000.0 - ef, e2_fno=ef, eps=e)
    if k == "truncate":
        on, no, _ = _exact_truncate(_density_matrix(c["nvir"], seed), c["po"])
        return dict(on=on, no=no * on, nkept=None)
    st = prepare(case, seed)
    if k == "ladder":
        b, t, nv = st["B"], st["T"], c["nv"]
        out = torch.empty_like(t)
        for a in range(nv):
            i = b[:, a, :].T @ b.reshape(-1, nv * nv)                       # [c][(b d)]
            i = i.reshape(nv, nv, nv).transpose(0, 1).reshape(nv, nv * nv)  # [b][(c d)]
            out[:, a, :] = t.reshape(-1, nv * nv) @ i.T
        return dict(c=out)
    if k == "naf":
        b = st["B"].reshape(c["naux"], -1)
        w, u = torch.linalg.eigh(b @ b.T)
        w, u = w.flip(0), u.flip(1)
        top = u.gather(0, u.abs().argmax(0, keepdim=True))
        u = u * torch.where(top < 0, -1.0, 1.0)
        n = int((w > st["thr"]).sum())
        out = torch.zeros_like(b)
        out[:n] = u[:, :n].T @ b
        return dict(naux=None, w=w, b=out.reshape(c["naux"], c["nh"], c["np"]))
    ms = _batch_members(c)
    if work(case)["flops"] > 8e12:
        return None
    out = [_exact_step(m, _molecule(m, seed * 100 + i), c["po"]) for i, m in enumerate(ms)]
    return dict(e2=[o["e2"] for o in out], nkept=[None for _ in out], de=[o["de"] for o in out], d=[o["d"] for o in out],
                on=[o["on"] for o in out])
