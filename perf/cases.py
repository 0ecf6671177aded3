"""What a self-consistent GW program spends its time on, as calls of this package.

A run of the method repeats five steps on one system: the static self-energy
(`hf`), the polarization P~0 (`polarization`), the screened solve (`screened`),
the self-energy (`selfenergy`) and the Dyson equation with its
chemical-potential search (`dyson`).  A program calls them one by one, as
`iterate`, or for many small systems at once as `batch_iterate`; a gradient-based
one goes through the `torch.autograd` functions.  The cases below are these calls
at the sizes of this repository's workloads: the toy solid (nao 8, naux 32), the
silicon-sized system (26, 200, 92 tau points), the large system (52, 400, 100), and
the members of the uneven batch (nao 8 to 40, naux = 8 nao, 64 tau points).  The
large and silicon-sized systems run on smaller k-meshes than 4x4x4 and 3x3x3, so
that a pass stays below a second; the work per (q, k) pair is that of the full mesh.

Inputs follow the package's synthetic systems: H0 with a spectrum in [-1, 1] Ha,
S near the identity, V^{kk'}(Q) Gaussian with magnitude exp(-Q/8) and the pairing
V^{k'k}(Q) = V^{kk'}(Q)^H, G(tau) the non-interacting Green's function of (H0, S),
and P~0(i Omega), P~(tau) sums of bosonic poles with positive residues, which have
the symmetries of a polarization: Hermitian in tau, and the value at -q and beta - tau
is the complex conjugate.

The mixed-precision paths multiply in pieces of 22 (16) bits and accumulate in FP32:
what they compute has single precision whatever the width of the buffer, and a
program keeps it as complex64 (P~ of the large system is then 8 GB instead of 16).
`run` hands those results over that way; the FP64 path's stay complex128.
"""
import math

import numpy as np
import torch

from paper_2206_07660_gb300 import GW
from paper_2206_07660_gb300.autograd import Polarization, SelfEnergy
from paper_2206_07660_gb300.gw import batch_iterate

MIXED = ("split_f16", "split_tf32", "split_bf16", "fp32")


def listed():
    return [
        # The smallest call: one iteration of the toy solid in FP64, launches and host work.
        dict(name="iterate_toy_fp64", kind="iterate", precision="fp64", nao=8, naux=32, mesh="2x2x2", ntau=32,
             beta=100.0),
        # A screening campaign: four systems of the uneven batch, one captured iteration of each.
        dict(name="batch_uneven_f16", kind="batch", precision="split_f16", systems="8:64:3x3x3 12:96:2x2x2 "
             "16:128:2x2x2 26:208:2x2x1", ntau=64, beta=100.0),
        # The two contractions of the large system on the benchmark's mixed path.
        dict(name="polarization_large_f16", kind="polarization", precision="split_f16", nao=52, naux=400,
             mesh="2x2x1", ntau=100, beta=1000.0),
        dict(name="selfenergy_large_f16", kind="selfenergy", precision="split_f16", nao=52, naux=400, mesh="2x2x1",
             ntau=100, beta=1000.0),
        # The screened solve between them (FP64 accuracy), 400 matrices of order 400.
        dict(name="screened_large", kind="screened", precision="split_f16", nao=52, naux=400, mesh="2x2x1", ntau=100,
             beta=1000.0),
        # Members of the uneven batch by themselves: many (q, k) pairs with little work in each.
        dict(name="polarization_small_f16", kind="polarization", precision="split_f16", nao=8, naux=64, mesh="4x4x4",
             ntau=64, beta=100.0),
        dict(name="selfenergy_middle_f16", kind="selfenergy", precision="split_f16", nao=16, naux=128, mesh="3x3x3",
             ntau=64, beta=100.0),
        # The silicon-sized system: FP64, the other split of the mixed path, a mesh with q != -q.
        dict(name="polarization_silicon_fp64", kind="polarization", precision="fp64", nao=26, naux=200, mesh="3x1x1",
             ntau=92, beta=1000.0),
        dict(name="selfenergy_silicon_tf32", kind="selfenergy", precision="split_tf32", nao=26, naux=200,
             mesh="3x2x1", ntau=92, beta=1000.0),
        # Gradients through the two contractions: FP64, and complex64 arithmetic.
        dict(name="gradient_polarization_fp64", kind="grad_polarization", precision="fp64", nao=26, naux=200,
             mesh="2x1x1", ntau=92, beta=1000.0),
        dict(name="gradient_selfenergy_c64", kind="grad_selfenergy", precision="split_f16", nao=26, naux=200,
             mesh="2x2x1", ntau=92, beta=1000.0),
        # The steps between two self-energies: Hartree-Fock, then Dyson with the mu search.
        dict(name="hf_dyson_large", kind="hf_dyson", precision="split_f16", nao=52, naux=400, mesh="2x2x2", ntau=100,
             beta=1000.0),
    ]


# What a drawn case may cost, as the listed ones of its kind and arithmetic do (see `work`).
_LIMIT = {"fp64": 9e10, "fp32": 1.5e12, "split_tf32": 2.5e12, "split_bf16": 4.2e12, "split_f16": 4.2e12}
_MESHES = ("1x1x1", "2x1x1", "3x1x1", "2x2x1", "3x2x1", "4x2x1", "2x2x2", "3x3x1", "3x2x2", "5x2x1", "3x3x3", "4x3x2",
           "4x4x2", "4x4x4")


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(("iterate", "batch", "polarization", "polarization", "selfenergy", "selfenergy", "screened",
                           "grad_polarization", "grad_selfenergy", "hf_dyson"))
        precision = rng.choice(("fp64", "split_f16", "split_f16", "split_f16", "split_tf32", "split_bf16", "fp32"))
        beta = rng.choice((100.0, 1000.0)) if kind != "batch" else 100.0
        ntau = rng.randint(64, 100) if beta > 500 else rng.randint(32, 72)
        if kind == "batch":
            if precision not in ("fp64", "split_f16"):
                continue
            one = []
            for _ in range(rng.randint(2, 4)):
                nao = rng.choice((8, 9, 12, 13, 16, 26))
                one.append("%d:%d:%s" % (nao, nao * rng.randint(3, 8), rng.choice(_MESHES[1:8])))
            case = dict(kind=kind, precision=precision, systems=" ".join(one), ntau=max(ntau, 48), beta=beta)
        else:
            nao = _log(rng, 4, 52)
            case = dict(kind=kind, precision=precision, nao=nao, naux=min(400, int(nao * rng.uniform(3, 10))),
                        mesh=rng.choice(_MESHES), ntau=ntau, beta=beta)
            if kind == "iterate" and (precision != "fp64" or ntau < 48):
                continue
        # a Dyson solution wants a level near mu: enough levels for the temperature
        if kind in ("iterate", "batch", "hf_dyson") and \
                min(m["nao"] * _mesh(m)[1] for m in (_members(case) if kind == "batch" else [case])) < 0.5 * beta:
            continue
        w = work(case)
        # the gradient of P~0 runs in FP64 on every path, that of Sigma~ in complex64 on the mixed ones
        limit = _LIMIT["fp64" if kind == "grad_polarization" else precision]
        if kind == "grad_selfenergy" and precision != "fp64":
            limit = 9e11
        if kind in ("screened", "hf_dyson"):
            limit = 1.2e11
        if w["flops"] <= limit and w["bytes"] <= 4e9:
            return case


# ---------------------------------------------------------------- sizes

def _mesh(case):
    n = [int(x) for x in case["mesh"].split("x")]
    return n, n[0] * n[1] * n[2]


def _members(case):
    out = []
    for s in case["systems"].split():
        nao, naux, mesh = s.split(":")
        out.append(dict(nao=int(nao), naux=int(naux), mesh=mesh, ntau=case["ntau"], beta=case["beta"]))
    return out


def work(case):
    """Bytes: inputs once and outputs once.  Flops: 8 per complex multiply-add of the contractions as
    products of three factors, each pair of values that are complex conjugates of one another once
    ((q, tau) with (-q, beta - tau) in the contractions, Q with Q' in P~0), and n^3 multiply-adds per
    screened system."""
    if case["kind"] == "batch":
        parts = [work(dict(m, kind="iterate", precision=case["precision"])) for m in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    _, nk = _mesh(case)
    nao, naux, nt = case["nao"], case["naux"], case["ntau"]
    v, g, p = 16.0 * nk * nk * naux * nao * nao, 16.0 * nt * nk * nao * nao, 16.0 * nk * nt * naux * naux
    k = 16.0 * nk * nao * nao
    outer, inner = 8.0 * nt * nk * nk * naux * naux * nao * nao, 8.0 * nt * nk * nk * naux * nao ** 3
    f_pol, f_sig = outer / 4 + inner, outer / 2 + 2 * inner
    f_scr = 8.0 * nk * nt * naux ** 3 / 2
    f_hf = 16.0 * nk * nk * naux * nao ** 3 / 2 + 32.0 * nk * naux * nao * nao
    f_dys = 8.0 * nk * nt * nao ** 3 * 12
    return {"polarization": dict(bytes=v / 2 + g + p, flops=f_pol),
            "selfenergy": dict(bytes=v / 2 + 2 * g + p, flops=f_sig),
            "screened": dict(bytes=3 * p, flops=f_scr),
            "grad_polarization": dict(bytes=v / 2 + 2 * g + 2 * p, flops=3 * f_pol),
            "grad_selfenergy": dict(bytes=v / 2 + 4 * g + 2 * p, flops=3 * f_sig),
            "hf_dyson": dict(bytes=v + 4 * g + 4 * k, flops=f_hf + f_dys),
            "iterate": dict(bytes=v + 4 * g + 2 * p, flops=f_pol + f_sig + f_scr + f_hf + f_dys)}[case["kind"]]


# ---------------------------------------------------------------- inputs

def _indices(ntau):
    """Sampled fermionic and bosonic Matsubara integers: consecutive at first, then spreading as a tangent."""
    def positive(h):
        raw = np.floor(0.4 * h * np.tan(np.pi * (np.arange(h) + 0.5) / (2 * (h + 1))))
        out, prev = [], -1
        for x in raw:
            prev = max(int(x), prev + 1)
            out.append(prev)
        return np.array(out, dtype=np.int64)
    hf, hb = (ntau + 1) // 2, ntau // 2
    p, pb = positive(hf), positive(hb) + 1
    fermi = np.sort(np.concatenate([p, -p[:ntau - hf] - 1]))
    bose = np.sort(np.concatenate([[0], pb, -pb[:ntau - 1 - hb]]))
    return fermi, bose


def _tau(beta, ntau):
    return 0.5 * beta * (1.0 - np.cos(np.pi * (2 * np.arange(ntau) + 1) / (2 * ntau)))


def _cn(gen, *shape):
    return torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=gen)


def _herm(x):
    return 0.5 * (x + x.mH)


def _minus(mesh):
    n1, n2, n3 = mesh
    return torch.tensor([((-a % n1) * n2 + (-b % n2)) * n3 + (-c % n3)
                         for a in range(n1) for b in range(n2) for c in range(n3)], device="cuda")


def _system(case, seed):
    """H0, S, V and the non-interacting G(tau), on the GPU."""
    mesh, nk = _mesh(case)
    nao, naux, nt, beta = case["nao"], case["naux"], case["ntau"], case["beta"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    U = torch.linalg.qr(_cn(gen, nk, nao, nao))[0]
    e = 2.0 * torch.rand(nk, nao, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    H0 = _herm((U * e[:, None, :].to(U.dtype)) @ U.mH)
    S = torch.eye(nao, dtype=torch.complex128, device="cuda") + 0.05 * _herm(_cn(gen, nk, nao, nao)) / math.sqrt(nao)
    decay = torch.exp(-torch.arange(naux, dtype=torch.float64, device="cuda") / 8.0) * 0.35 / math.sqrt(nao)
    V = _cn(gen, nk, nk, naux, nao, nao) * decay[:, None, None]
    for k in range(nk):
        V[k, k] = (V[k, k] + V[k, k].mH) / math.sqrt(2.0)
        if k:
            V[k, :k] = V[:k, k].mH
    return dict(mesh=mesh, nk=nk, H0=H0.contiguous(), S=S.contiguous(), V=V, gen=gen)


def _green(case, s):
    """G(tau) = -sum_n c_n c_n^H e^{-e_n tau} (1 - f(e_n)) of H0 c = e S c at mu = 0."""
    tau = torch.from_numpy(_tau(case["beta"], case["ntau"])).cuda()
    L = torch.linalg.cholesky(s["S"])
    X = torch.linalg.solve_triangular(L, s["H0"], upper=False)
    X = torch.linalg.solve_triangular(L, X.mH, upper=False)
    e, C = torch.linalg.eigh(_herm(X))
    C = torch.linalg.solve_triangular(L.mH, C, upper=True)
    t = tau[:, None, None]
    w = torch.exp(-torch.where(e > 0, e * t, -e * (case["beta"] - t))) / (1.0 + torch.exp(-case["beta"] * e.abs()))
    G = -(C[None] * w[:, :, None, :].to(C.dtype)) @ C.mH[None]
    return _herm(G).contiguous()


def _residues(case, s, poles, scale):
    """Positive residues A_r^q = u u^H of `poles` poles, decaying with Q as V does."""
    naux, nk = case["naux"], s["nk"]
    decay = torch.exp(-torch.arange(naux, dtype=torch.float64, device="cuda") / 8.0)
    u = _cn(s["gen"], poles, nk, naux, max(2, naux // 8)) * decay[:, None] * math.sqrt(scale / max(2, naux // 8))
    return u @ u.mH


def _boson_tau(case, s):
    """P~^q(tau) = -sum_r (A_r^q e^{-w tau} + conj A_r^{-q} e^{-w (beta - tau)}) / (1 - e^{-beta w})."""
    beta, neg = case["beta"], _minus(s["mesh"])
    tau = torch.from_numpy(_tau(beta, case["ntau"])).cuda()
    P = torch.zeros(s["nk"], case["ntau"], case["naux"], case["naux"], dtype=torch.complex128, device="cuda")
    for w, A in zip((0.4, 1.1, 2.3), _residues(case, s, 3, 0.5)):
        a = torch.exp(-w * tau) / (1.0 - math.exp(-beta * w))
        P -= A[:, None] * a[:, None, None]
    P += P[neg].flip(1).conj()
    return _herm(P).contiguous()


def _boson_iw(case, s):
    """P~0^q(i Omega) = -sum_r (A_r^q / (w - i Omega) + conj A_r^{-q} / (w + i Omega))."""
    om = torch.from_numpy(2.0 * np.pi / case["beta"] * _indices(case["ntau"])[1]).cuda()
    P = torch.zeros(s["nk"], case["ntau"], case["naux"], case["naux"], dtype=torch.complex128, device="cuda")
    for w, A in zip((0.4, 1.1, 2.3), _residues(case, s, 3, 2.0)):
        P -= A[:, None] / torch.complex(torch.full_like(om, w), -om)[:, None, None]
    return (P + P[_minus(s["mesh"])].conj()).contiguous()


def _context(case, s, **more):
    fn, bm = _indices(case["ntau"])
    return GW(s["H0"], s["S"], s["V"], s["mesh"], case["ntau"], case["beta"], fn, bm, n_elec=case["nao"],
              precision=case["precision"], borrow_V=True, **more)


def _like(gw, name):
    return torch.empty(gw.shape_of(name), dtype=torch.complex128, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        one = [prepare(dict(m, kind="iterate", precision=case["precision"]), seed * 31 + i)
               for i, m in enumerate(_members(case))]
        batch_iterate([o["gw"] for o in one], 2)    # captures the graphs, as the first iterations of a campaign do
        return dict(kind=kind, one=one, single=case["precision"] in MIXED)
    s = _system(case, seed)
    single = case["precision"] in MIXED
    st = dict(kind=kind, single=single, V=s["V"])
    st["gw"] = gw = _context(case, s, damping=1.0 if kind.startswith(("self", "grad")) else 0.5)
    if kind == "screened":
        st["P0_iw"] = _boson_iw(case, s)
        st["P_iw"], st["P_tau"] = _like(gw, "P_iw"), _like(gw, "P_tau")
        return st
    st["G"] = _green(case, s)
    if kind in ("selfenergy", "grad_selfenergy"):
        st["P"] = _boson_tau(case, s)
    if kind == "grad_polarization":
        st["bar"] = _cn(s["gen"], *gw.shape_of("P0_tau"))
    if kind == "grad_selfenergy":
        st["bar"] = _cn(s["gen"], *gw.shape_of("Sigma_tau"))
        gw.adjoint_c64 = case["precision"] in MIXED
    if kind == "polarization":
        st["out"] = _like(gw, "P0_tau")
    if kind == "selfenergy":
        st["out"] = _like(gw, "Sigma_tau")
    if kind in ("iterate", "hf_dyson"):
        # a self-energy to start from: a static part and poles at +-1 Ha with positive residues
        nk, nao = s["nk"], case["nao"]
        st["Sinf"] = (0.02 * _herm(_cn(s["gen"], nk, nao, nao)) / math.sqrt(nao)).contiguous()
        wn = torch.from_numpy((2 * _indices(case["ntau"])[0] + 1) * np.pi / case["beta"]).cuda()
        Siw = torch.zeros(gw.shape_of("Sigma_iw"), dtype=torch.complex128, device="cuda")
        for e in (-1.0, 1.0):
            u = _cn(s["gen"], nk, nao, nao) * (0.1 / math.sqrt(nao))
            Siw += (u @ u.mH)[None] / torch.complex(torch.full_like(wn, -e), wn)[:, None, None, None]
        st["Siw"] = Siw
        for name in ("G_tau", "Sigma_inf", "Sigma_iw", "Sigma_inf_new"):
            st[name] = _like(gw, name)
    return st


# ---------------------------------------------------------------- passes

def _kept(x, single):
    """A result as the program keeps it: complex64 where the products have single precision."""
    return x.to(torch.complex64) if single else x


def _start(st):
    gw = st["gw"]
    gw.set("mu", 0.0)
    gw.set("G_tau", st["G"])
    gw.set("Sigma_inf", st["Sinf"])
    gw.set("Sigma_iw", st["Siw"])


def _state(st, single):
    gw = st["gw"]
    return {n: _kept(gw.get(n, out=st[n]), single) for n in ("G_tau", "Sigma_inf", "Sigma_iw")}


def run(state):
    kind, single = state["kind"], state["single"]
    if kind == "batch":
        for o in state["one"]:
            _start(o)
        batch_iterate([o["gw"] for o in state["one"]], 1)
        return [_state(o, single) for o in state["one"]]
    gw = state["gw"]
    if kind == "iterate":
        _start(state)
        gw.iterate(1)
        return _state(state, single)
    if kind == "polarization":
        gw.set("G_tau", state["G"])
        gw.polarization()
        return _kept(gw.get("P0_tau", out=state["out"]), single)
    if kind == "selfenergy":
        gw.set("G_tau", state["G"])
        gw.set("P_tau", state["P"])
        gw.selfenergy_partial()
        return _kept(gw.get("Sigma_tau", out=state["out"]), single)
    if kind == "screened":
        gw.set("P0_iw", state["P0_iw"])
        gw.screened()
        return {n: gw.get(n, out=state[n]) for n in ("P_iw", "P_tau")}
    if kind == "grad_polarization":
        G = state["G"].detach().requires_grad_(True)
        P0 = Polarization.apply(G, gw)
        P0.backward(state["bar"])
        return [_kept(P0.detach(), single), G.grad]
    if kind == "grad_selfenergy":
        G, P = (state[n].detach().requires_grad_(True) for n in ("G", "P"))
        Sig = SelfEnergy.apply(G, P, gw)
        Sig.backward(state["bar"])
        return [_kept(x, single) for x in (Sig.detach(), G.grad, P.grad)]
    _start(state)
    gw.hf()
    gw.dyson()
    return {"Sigma_inf_new": _kept(gw.get("Sigma_inf_new", out=state["Sigma_inf_new"]), single),
            "G_tau": gw.get("G_tau", out=state["G_tau"]), "mu": gw.get("mu")}


# ---------------------------------------------------------------- the same in 64 bits

def _pairs(mesh):
    n1, n2, n3 = mesh
    v = [(a, b, c) for a in range(n1) for b in range(n2) for c in range(n3)]
    at = {x: i for i, x in enumerate(v)}
    for q, vq in enumerate(v):
        for k, vk in enumerate(v):
            yield q, k, at[tuple((x + y) % n for x, y, n in zip(vk, vq, mesh))]


def _polarization64(case, s, G, bar=None):
    """P~0^q(tau)_QQ' = (2/Nk) sum_k tr[V^{k,k+q}(Q) G^{k+q}(tau) V^{k+q,k}(Q') G^k(-tau)], symmetrised;
    with `bar` also the gradient of Re <bar, P~0> with respect to G."""
    nk, nao, naux, nt = s["nk"], case["nao"], case["naux"], case["ntau"]
    V, Gm = s["V"], -G.flip(0)
    out = torch.zeros(nk, nt, naux, naux, dtype=torch.complex128, device="cuda")
    dG, dGm = torch.zeros_like(G), torch.zeros_like(G)
    hb = None if bar is None else _herm(bar) * (2.0 / nk)
    for q, k, kq in _pairs(s["mesh"]):
        A = V[k, kq]                                                      # [Q, d, a]
        B = V[kq, k].permute(2, 1, 0).reshape(nao * nao, naux)            # [(c, b), Q'] = V_bc(Q')
        Y = torch.matmul(A[None], G[:, kq][:, None])                      # [t, Q, d, b]
        Z = torch.matmul(Gm[:, k][:, None], Y)                            # [t, Q, c, b]
        out[q] += (Z.reshape(nt * naux, nao * nao) @ B).reshape(nt, naux, naux)
        if bar is not None:
            Zb = (hb[q].reshape(nt * naux, naux) @ B.mH).reshape(nt, naux, nao, nao)
            dGm[:, k] += torch.einsum("tqcb,tqdb->tcd", Zb, Y.conj())
            Yb = torch.matmul(Gm[:, k].mH[:, None], Zb)
            dG[:, kq] += torch.einsum("qda,tqdb->tab", A.conj(), Yb)
    P0 = _herm(out * (2.0 / nk))
    return (P0, None) if bar is None else (P0, dG - dGm.flip(0))


def _selfenergy64(case, s, G, P, bar=None):
    """Sigma~^k(tau) = -(1/Nk) sum V^{k,k-q}(Q) G^{k-q}(tau) P~^q_QQ'(tau) V^{k-q,k}(Q'), symmetrised, and
    the gradients of Re <bar, Sigma~> with respect to G and P~."""
    nk, nao, naux, nt = s["nk"], case["nao"], case["naux"], case["ntau"]
    V, out = s["V"], torch.zeros_like(G)
    dG, dP = torch.zeros_like(G), None if bar is None else torch.zeros_like(P)
    hb = None if bar is None else _herm(bar) * (-1.0 / nk)
    for q, kmq, k in _pairs(s["mesh"]):                                   # k = kmq + q
        A = V[k, kmq].reshape(naux, nao * nao)                            # [Q, (i, a)]
        W = V[kmq, k].reshape(naux * nao, nao)                            # [(Q', b), j]
        X = torch.matmul(P[q].transpose(1, 2), A[None]).reshape(nt, naux, nao, nao)      # [t, Q', i, a]
        Y = torch.matmul(X, G[:, kmq][:, None])                           # [t, Q', i, b]
        out[:, k] += Y.transpose(1, 2).reshape(nt, nao, naux * nao) @ W
        if bar is not None:
            Yb = (hb[:, k] @ W.mH).reshape(nt, nao, naux, nao).transpose(1, 2)
            dG[:, kmq] += torch.einsum("tqia,tqib->tab", X.conj(), Yb)
            Xb = torch.matmul(Yb, G[:, kmq].mH[:, None]).reshape(nt, naux, nao * nao)
            dP[q] += torch.matmul(Xb, A.mH[None]).transpose(1, 2)
    return _herm(out * (-1.0 / nk)), dG, dP


def _density64(case, G):
    """gamma = -G(beta^-) of the polynomial through the Chebyshev nodes."""
    nt = case["ntau"]
    j, k = np.arange(nt), np.arange(nt)[:, None]
    C = (2.0 / nt) * np.cos(k * np.arccos(-np.cos(np.pi * (2 * j + 1) / (2 * nt)))[None, :])
    C[0] = 1.0 / nt
    return -torch.einsum("j,jkab->kab", torch.from_numpy(C.sum(0)).cuda().to(G.dtype), G)


def _static64(case, s, G):
    """Hartree and exchange of the density matrix."""
    nk, nao, naux, V = s["nk"], case["nao"], case["naux"], s["V"]
    g = _density64(case, G)
    D = torch.stack([V[k, k] for k in range(nk)])
    out = (2.0 / nk) * torch.einsum("kqij,q->kij", D, torch.einsum("kab,kqba->q", g, D))
    for k in range(nk):
        for p in range(nk):
            Y = torch.matmul(V[k, p], g[p]).transpose(0, 1).reshape(nao, naux * nao)
            out[k] -= Y @ V[p, k].reshape(naux * nao, nao) / nk
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("iterate", "batch") or work(case)["flops"] > 6e12:
        return None
    s = _system(case, seed)
    if kind == "screened":
        P0 = _boson_iw(case, s)
        eye = torch.eye(case["naux"], dtype=torch.complex128, device="cuda")
        return {"P_iw": torch.stack([torch.linalg.solve(eye - p, p) for p in P0]), "P_tau": None}
    G = _green(case, s)
    if kind == "polarization":
        return _polarization64(case, s, G)[0]
    if kind == "grad_polarization":
        bar = _cn(s["gen"], s["nk"], case["ntau"], case["naux"], case["naux"])
        return list(_polarization64(case, s, G, bar))
    if kind == "selfenergy":
        return _selfenergy64(case, s, G, _boson_tau(case, s))[0]
    if kind == "grad_selfenergy":
        P = _boson_tau(case, s)
        return list(_selfenergy64(case, s, G, P, _cn(s["gen"], case["ntau"], s["nk"], case["nao"], case["nao"])))
    return {"Sigma_inf_new": _static64(case, s, G), "G_tau": None, "mu": None}
