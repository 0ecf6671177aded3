"""Routes that the stage tests at small sizes do not reach: the FP64 digit products under the tangents, for a V
that does not fold, with operands longer than their workspace, and GW_TRS at odd orbital counts on the 16-bit
splits."""
import numpy as np
import pytest

from gpu_helpers import gpu, hermitian_noise, rel, system
from oracle import adjoint as oad
from oracle import gw as ogw

pytestmark = pytest.mark.gpu

TOL = 1e-12   # FP64 sums of ~1e3 products of order one


def _noise(*shape):
    rng = np.random.default_rng(sum(shape))
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _dev(x):
    import torch
    return torch.from_numpy(x).cuda()


@pytest.mark.parametrize("loose", [False, True])
def test_tangents_and_adjoints_in_digits(loose):
    nao, naux, kmesh, ntau = 17, 75, (3, 1, 1), 40
    sysd = system(nao, naux, kmesh, ntau, 20.0, 181)
    km = ogw.KMesh(kmesh)
    if loose:   # accepted, but beyond the pairing that the folds ask for
        sysd["V"] = sysd["V"] * (1.0 + 1e-13 * np.random.default_rng(182).standard_normal(sysd["V"].shape))
    tol = 1e-11 if loose else TOL   # (the adjoint chains take one of the two sides of the pairing)
    V, qs = sysd["V"], list(range(km.nk))
    G, P = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 183), hermitian_noise((km.nk, ntau, naux, naux), 0.3, 184)
    dG, dP = _noise(*G.shape), _noise(*P.shape)
    g = gpu(sysd)
    g.set("G_tau", G)
    g.set("P_tau", P)
    ref = 0.5 * (ogw.polarization_tau(V, G + dG, km) - ogw.polarization_tau(V, G - dG, km))
    assert rel(g.polarization_jvp(_dev(dG)).cpu().numpy(), ref) < tol
    ref = ogw.selfenergy_tau(V, dG, P, km, qs=qs) + ogw.selfenergy_tau(V, G, dP, km, qs=qs)
    assert rel(g.selfenergy_jvp(_dev(dG), _dev(dP)).cpu().numpy(), ref) < tol
    assert rel(g.polarization_vjp(_dev(dP)).cpu().numpy(), oad.polarization_vjp(V, G, km, dP)) < tol
    gb, pb = g.selfenergy_vjp(_dev(dG))
    rg, rp = oad.selfenergy_vjp(V, G, P, km, dG)
    assert rel(gb.cpu().numpy(), rg) < tol and rel(pb.cpu().numpy(), rp) < tol


@pytest.mark.parametrize("nao,naux,ntau", [(40, 300, 80), (5, 400, 216)])
def test_operands_longer_than_their_workspace(nao, naux, ntau):
    # digits of more than 1 GB: rows, tau points and batch entries in pieces; native FP64 arithmetic as the other side
    sysd = system(nao, naux, (1, 1, 1), ntau, 20.0, 185)
    G, P = hermitian_noise((ntau, 1, nao, nao), 0.3, 186), hermitian_noise((1, ntau, naux, naux), 0.3, 187)
    Pbar, Sbar = _dev(_noise(1, ntau, naux, naux)), _dev(_noise(ntau, 1, nao, nao))
    out = []
    for arith in ("tensor", "native"):
        g = gpu(sysd, fp64_gemm=arith)
        g.set("G_tau", G)
        g.polarization()
        r = [g.get("P0_tau"), g.polarization_vjp(Pbar).cpu().numpy()]
        g.set("P_tau", P)
        g.selfenergy_partial()
        r += [g.get("Sigma_tau")] + [x.cpu().numpy() for x in g.selfenergy_vjp(Sbar)]
        out.append(r)
        g.close()
    for a, b in zip(*out):
        assert rel(a, b) < TOL


@pytest.mark.parametrize("nao", [3, 7, 9, 13, 16, 17, 21])
@pytest.mark.parametrize("kmesh", [(3, 2, 1), (2, 2, 1)])
@pytest.mark.parametrize("precision,tol", [("fp64", TOL), ("split_f16", 5e-6), ("split_bf16", 5e-5)])
def test_trs_at_any_orbital_count(nao, kmesh, precision, tol):
    naux, ntau = 23, 13
    sysd = system(nao, naux, kmesh, ntau, 20.0, 188, trs=True)
    km = ogw.KMesh(kmesh)
    neg = [km.index(-km.vec[k]) for k in range(km.nk)]
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.05, 189) - 0.3 * np.eye(nao)
    G = 0.5 * (G + np.conj(G[:, neg]))
    g = gpu(sysd, precision=precision, trs=True)
    g.set("G_tau", G)
    g.polarization()
    assert rel(g.get("P0_tau"), ogw.polarization_tau(sysd["V"], G, km)) < tol
    g.screened()
    P = g.get("P_tau")
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau"), ogw.selfenergy_tau(sysd["V"], G, P, km, qs=list(range(km.nk)))) < tol
    # a P~ that is handed in, with time-reversal symmetry alone
    P = hermitian_noise((km.nk, ntau, naux, naux), 0.3, 190)
    P = 0.5 * (P + np.conj(P[neg]))
    g.set("P_tau", P)
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau"), ogw.selfenergy_tau(sysd["V"], G, P, km, qs=list(range(km.nk)))) < tol


def test_fp64_stages_in_a_callers_capture():
    # digit products, their range check and the tiles left to FP64 arithmetic, replayed on level and graded G
    import torch
    nao, naux, kmesh, ntau = 17, 75, (3, 1, 1), 40
    sysd = system(nao, naux, kmesh, ntau, 20.0, 191)
    km = ogw.KMesh(kmesh)
    G, P = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 192), hermitian_noise((km.nk, ntau, naux, naux), 0.3, 193)
    s = 2.0 ** np.random.default_rng(194).permutation(np.round(np.linspace(-10, 10, nao)))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        g = gpu(sysd)
        g.set("G_tau", hermitian_noise(G.shape, 0.3, 195))
        graphs = []
        for stage in (g.polarization, g.selfenergy_partial):
            g.set("P_tau", P)
            stage()
            torch.cuda.synchronize()
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[-1], stream=stream):
                stage()
            g.set("P_tau", P)
        for X in (G, G / np.outer(s, s)):
            g.set("G_tau", X)
            graphs[0].replay()
            torch.cuda.synchronize()
            assert rel(g.get("P0_tau"), ogw.polarization_tau(sysd["V"], X, km)) < TOL
            g.set("P_tau", P)
            graphs[1].replay()
            torch.cuda.synchronize()
            assert rel(g.get("Sigma_tau"), ogw.selfenergy_tau(sysd["V"], X, P, km, qs=list(range(km.nk)))) < TOL
