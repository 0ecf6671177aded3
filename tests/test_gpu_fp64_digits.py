"""The large products of the FP64 contraction chains in digits on the tensor cores (the default of
FP64-accurate arithmetic) against the oracle: the last P~0 step, the first Sigma~ step, and those of
the two adjoints.  Sizes above the rule's 2e8 flops with odd orders, K longer and shorter than one
exact range (and one whose first P~0 step takes the digits for a part of the q), native FP64 arithmetic
as the other side, and values that are not finite."""
import numpy as np
import pytest

from gpu_helpers import gpu, hermitian_noise, rel, system
from oracle import adjoint as oad
from oracle import gw as ogw

pytestmark = pytest.mark.gpu

# sums of ~1e3 products of order one: 2^-53 sqrt(1e3) per term of the largest sum, with margin
TOL = 1e-12
SIZES = [(13, 97, (2, 1, 1), 41), (17, 75, (3, 1, 1), 40), (5, 200, (1, 1, 1), 50), (21, 80, (3, 1, 1), 40)]


@pytest.mark.parametrize("nao,naux,kmesh,ntau", SIZES)
@pytest.mark.parametrize("arith", ["tensor", "native"])
def test_contractions(nao, naux, kmesh, ntau, arith):
    sysd = system(nao, naux, kmesh, ntau, 20.0, 101)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 102)
    P = hermitian_noise((km.nk, ntau, naux, naux), 0.3, 103)
    g = gpu(sysd, fp64_gemm=arith)
    g.set("G_tau", G)
    g.polarization()
    assert rel(g.get("P0_tau"), ogw.polarization_tau(sysd["V"], G, km)) < TOL
    g.set("P_tau", P)
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau"), ogw.selfenergy_tau(sysd["V"], G, P, km, qs=list(range(km.nk)))) < TOL


@pytest.mark.parametrize("nao,naux,kmesh,ntau", SIZES[:2])
@pytest.mark.parametrize("precision", ["fp64", "split_f16"])
def test_adjoints(nao, naux, kmesh, ntau, precision):
    import torch
    sysd = system(nao, naux, kmesh, ntau, 20.0, 104)
    km = ogw.KMesh(kmesh)
    rng = np.random.default_rng(105)
    noise = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    G, P = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 106), hermitian_noise((km.nk, ntau, naux, naux), 0.3, 107)
    g = gpu(sysd, precision=precision)
    g.set("G_tau", G)
    g.set("P_tau", P)
    Pbar, Sbar = noise(km.nk, ntau, naux, naux), noise(ntau, km.nk, nao, nao)
    got = g.polarization_vjp(torch.from_numpy(Pbar).cuda()).cpu().numpy()
    assert rel(got, oad.polarization_vjp(sysd["V"], G, km, Pbar)) < TOL
    gb, pb = g.selfenergy_vjp(torch.from_numpy(Sbar).cuda())
    rg, rp = oad.selfenergy_vjp(sysd["V"], G, P, km, Sbar)
    assert rel(gb.cpu().numpy(), rg) < TOL and rel(pb.cpu().numpy(), rp) < TOL


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_values_that_are_not_finite_stay_so(value):
    nao, naux, kmesh, ntau = SIZES[2]
    sysd = system(nao, naux, kmesh, ntau, 20.0, 108)
    G = hermitian_noise((ntau, 1, nao, nao), 0.3, 109)
    G[3, 0, 2, 2] = value
    g = gpu(sysd)
    g.set("G_tau", G)
    g.polarization()
    P0 = g.get("P0_tau")[0]
    bad = [3, ntau - 1 - 3]
    assert not np.isfinite(P0[bad]).any()
    assert np.isfinite(np.delete(P0, bad, axis=0)).all()


@pytest.mark.parametrize("scale", [1e-146, 1e-200])
def test_products_near_the_smallest_number(scale):
    # rows whose product is 1e-292, or underflows: the number itself (the last bits of sums of 1e3 terms of
    # which those below 1e-308 are lost, 1e-16 of the largest), not one of the smallest scale
    nao, naux, kmesh, ntau = SIZES[0]
    sysd = system(nao, naux, kmesh, ntau, 20.0, 110)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 111) * scale
    g = gpu(sysd)
    g.set("G_tau", G)
    g.polarization()
    ref = ogw.polarization_tau(sysd["V"], G, km)
    T = ogw.State(sysd).grid.TFb
    for name, x in (("P0_tau", ref), ("P0_iw", ogw.to_matsubara(T, ref, 1))):
        assert np.abs(g.get(name) - x).max() <= 1e-12 * np.abs(x).max(), name


def _scales(n, seed):
    """Powers of two from 2^-13 to 2^13 in random order (exact, and 1e8 between the ends)."""
    return 2.0 ** np.random.default_rng(seed).permutation(np.round(np.linspace(-13, 13, n)))


@pytest.mark.parametrize("nao,naux,kmesh,ntau", [SIZES[0], SIZES[3]])
def test_orbitals_and_auxiliaries_of_different_scale(nao, naux, kmesh, ntau):
    # V carries the scales of both indices, G and P~ their inverses: FP64 arithmetic does not see them
    # (scaling by powers of two), and the results are the unscaled ones'
    import torch
    sysd = system(nao, naux, kmesh, ntau, 20.0, 112)
    km = ogw.KMesh(kmesh)
    G, P = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 113), hermitian_noise((km.nk, ntau, naux, naux), 0.3, 114)
    V = sysd["V"]
    rng = np.random.default_rng(115)
    noise = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    Pbar, Sbar = noise(km.nk, ntau, naux, naux), noise(ntau, km.nk, nao, nao)
    s, u = np.outer(*[_scales(nao, 116)] * 2), np.outer(*[_scales(naux, 117)] * 2)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    ref_p0 = ogw.polarization_tau(V, G, km)
    ref_pg = oad.polarization_vjp(V, G, km, Pbar)
    ref_s = ogw.selfenergy_tau(V, G, P, km, qs=list(range(km.nk)))
    ref_sg, ref_sp = oad.selfenergy_vjp(V, G, P, km, Sbar)
    g = gpu(dict(sysd, V=V * s))
    g.set("G_tau", G / s)
    g.polarization()
    assert rel(g.get("P0_tau"), ref_p0) < TOL
    assert rel(g.polarization_vjp(dev(Pbar)).cpu().numpy() / s, ref_pg) < TOL
    g = gpu(dict(sysd, V=V * s * np.sqrt(np.diag(u))[:, None, None]))
    g.set("G_tau", G / s)
    g.set("P_tau", P / u)
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau") / s, ref_s) < TOL
    gb, pb = g.selfenergy_vjp(dev(Sbar / s))
    assert rel(gb.cpu().numpy() / s, ref_sg) < TOL and rel(pb.cpu().numpy() / u, ref_sp) < TOL


def test_one_tau_point_of_another_scale():
    # one tau point and one auxiliary function graded: tiles in digits and in FP64 in one product
    nao, naux, kmesh, ntau = SIZES[3]
    sysd = system(nao, naux, kmesh, ntau, 20.0, 118)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 119)
    s = _scales(nao, 120)
    G[7] /= np.outer(s, s)
    G[ntau - 1 - 7] *= np.outer(s, s)
    V = sysd["V"].copy()
    V[:, :, 5] *= np.outer(s, s)
    g = gpu(dict(sysd, V=V))
    g.set("G_tau", G)
    g.polarization()
    got, ref = g.get("P0_tau"), ogw.polarization_tau(V, G, km)
    for t in (0, 7, 20, ntau - 1 - 7):
        for Q in (slice(0, 5), slice(5, 6), slice(6, None)):
            for R in (slice(0, 5), slice(5, 6), slice(6, None)):
                assert rel(got[:, t, Q, R], ref[:, t, Q, R]) < TOL, (t, Q, R)
