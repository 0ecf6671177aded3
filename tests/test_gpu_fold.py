"""The bosonic block folded by its symmetries.  P~0 folded over (q, tau) -> (-q, beta - tau): only half of the (q, tau) blocks are
contracted and the others are their conjugates.  Compared with the oracle, which
computes every block, over meshes whose q are their own negatives or come in pairs,
even and odd tau counts, parts of the q range, a G that is not Hermitian, and a V whose
pairing is too loose for the fold (the route over every block)."""
import numpy as np
import pytest

from gpu_helpers import gpu, hermitian_noise, rel, system
from oracle import gw as ogw

pytestmark = pytest.mark.gpu

# FP64 sums of ~1e3 terms; 22-bit pieces with FP32 accumulation (the tolerance of the
# stage tests), 16-bit pieces one power of 2^-6 coarser
TOL = {"fp64": 1e-12, "fp32": 5e-6, "split_tf32": 5e-6, "split_f16": 5e-6, "split_bf16": 5e-5}


@pytest.mark.parametrize("kmesh,ntau,qr", [((2, 2, 1), 10, None), ((2, 1, 1), 9, None), ((3, 1, 1), 8, None),
                                           ((3, 2, 1), 7, None), ((4, 1, 1), 6, (1, 3)), ((4, 1, 1), 5, (1, 4)),
                                           ((1, 1, 1), 1, None), ((1, 1, 1), 2, None)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "split_tf32", "split_f16", "split_bf16"])
def test_polarization_blocks(kmesh, ntau, qr, precision):
    sysd = system(5, 21, kmesh, ntau, 20.0, 71)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, 5, 5), 0.3, 72)
    qs = range(km.nk) if qr is None else range(*qr)
    ref = ogw.polarization_tau(sysd["V"], G, km, qs=list(qs))
    g = gpu(sysd, precision=precision)
    if qr is not None:
        g.set_q_range(*qr)
    g.set("G_tau", G)
    g.polarization()
    got = g.get("P0_tau")
    for q in qs:
        assert rel(got[q], ref[q]) < TOL[precision], q
    assert np.array_equal(got[list(qs)], np.conj(np.swapaxes(got[list(qs)], -1, -2)))


@pytest.mark.parametrize("nao", [1, 2, 4, 7, 8, 12, 13, 16])
@pytest.mark.parametrize("kmesh,ntau,naux", [((3, 1, 1), 5, 37), ((2, 1, 1), 4, 1), ((4, 2, 1), 3, 70)])
@pytest.mark.parametrize("precision", ["split_f16", "split_bf16"])
def test_polarization_of_few_orbitals(nao, kmesh, ntau, naux, precision):
    # both nao-sized steps in one FP32 kernel and every q of a kind in one launch
    sysd = system(nao, naux, kmesh, ntau, 20.0, 78)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 79)
    g = gpu(sysd, precision=precision)
    g.set("G_tau", G)
    g.polarization()
    got, ref = g.get("P0_tau"), ogw.polarization_tau(sysd["V"], G, km)
    for q in range(km.nk):
        assert rel(got[q], ref[q]) < TOL[precision], q


@pytest.mark.parametrize("kmesh,ntau", [((2, 1, 1), 7), ((3, 1, 1), 6)])
def test_polarization_of_any_g(kmesh, ntau):
    # the fold needs no symmetry of G: a complex G without any, FP64
    sysd = system(4, 13, kmesh, ntau, 20.0, 73)
    km = ogw.KMesh(kmesh)
    rng = np.random.default_rng(74)
    G = rng.standard_normal((ntau, km.nk, 4, 4)) + 1j * rng.standard_normal((ntau, km.nk, 4, 4))
    g = gpu(sysd)
    g.set("G_tau", G)
    g.polarization()
    assert rel(g.get("P0_tau"), ogw.polarization_tau(sysd["V"], G, km)) < TOL["fp64"]


@pytest.mark.parametrize("precision", ["fp64", "split_f16"])
def test_polarization_of_loosely_paired_v(precision):
    # a pairing defect of 1e-12 is accepted by the checks and takes the route over every block
    kmesh, ntau = (3, 1, 1), 6
    sysd = system(4, 13, kmesh, ntau, 20.0, 75)
    km = ogw.KMesh(kmesh)
    rng = np.random.default_rng(76)
    sysd["V"] = sysd["V"] * (1.0 + 1e-12 * rng.standard_normal(sysd["V"].shape))
    G = hermitian_noise((ntau, km.nk, 4, 4), 0.3, 77)
    g = gpu(sysd, precision=precision)
    g.set("G_tau", G)
    g.polarization()
    assert rel(g.get("P0_tau"), ogw.polarization_tau(sysd["V"], G, km)) < max(TOL[precision], 1e-11)


@pytest.mark.parametrize("kmesh,ntau,naux,qr", [((2, 2, 1), 16, 20, None), ((2, 1, 1), 15, 21, None),
                                                ((3, 1, 1), 16, 19, None), ((3, 2, 1), 13, 33, None),
                                                ((4, 1, 1), 14, 16, (1, 3)), ((4, 1, 1), 14, 17, (0, 4)),
                                                ((1, 1, 1), 12, 1, None)])
def test_screened_block(kmesh, ntau, naux, qr):
    # P~0(i Omega), P~(i Omega) and P~(tau) from P~0(tau): frequencies +-Omega and q-points +-q folded,
    # real matrices where q = -q (odd orders padded); FP64 accuracy of the refined solve, the last
    # transform amplifying rounding by the condition of the grid (~1e2 here)
    sysd = system(4, naux, kmesh, ntau, 20.0, 81)
    km = ogw.KMesh(kmesh)
    st = ogw.State(sysd)
    st.G_tau = -hermitian_noise((ntau, km.nk, 4, 4), 0.05, 82) - 0.3 * np.eye(4)
    st.sigma()
    g = gpu(sysd)
    if qr is not None:
        g.set_q_range(*qr)
    g.set("G_tau", st.G_tau)
    g.polarization()
    qs = list(range(km.nk) if qr is None else range(*qr))
    assert rel(g.get("P0_iw")[qs], st.P0_iw[qs]) < 1e-11
    g.screened()
    assert rel(g.get("P_iw")[qs], st.P_iw[qs]) < 1e-11
    assert rel(g.get("P_tau")[qs], st.P_tau[qs]) < 1e-10


@pytest.mark.parametrize("defect", [0.0, 1e-3])
def test_screened_of_a_given_p0(defect):
    # a P~0(i Omega) that is handed in is folded only when it has the symmetries
    kmesh, ntau, naux = (3, 2, 1), 14, 18
    sysd = system(4, naux, kmesh, ntau, 20.0, 83)
    km = ogw.KMesh(kmesh)
    st = ogw.State(sysd)
    st.G_tau = -hermitian_noise((ntau, km.nk, 4, 4), 0.05, 84) - 0.3 * np.eye(4)
    st.sigma()
    P0 = st.P0_iw + defect * hermitian_noise(st.P0_iw.shape, 1.0, 85)
    g = gpu(sysd)
    g.set("P0_iw", P0)
    g.screened()
    ref = ogw.screened(P0)
    assert rel(g.get("P_iw"), ref) < 1e-11
    assert rel(g.get("P_tau"), ogw.herm(ogw.to_matsubara(st.grid.TBb, ref, 1))) < 1e-10


def _folded(P, km):
    """P~ with the mirror symmetry P~^{-q}(beta - tau) = conj P~^q(tau), exactly."""
    neg = [km.index(-km.vec[q]) for q in range(km.nk)]
    return 0.5 * (P + np.conj(P[neg][:, ::-1]))


@pytest.mark.parametrize("nao,kmesh,ntau,qr", [(4, (2, 2, 1), 6, None), (5, (2, 1, 1), 5, None), (7, (3, 1, 1), 5, None),
                                               (13, (3, 2, 1), 4, None), (8, (4, 1, 1), 5, (1, 4)),
                                               (3, (4, 1, 1), 4, (1, 3)), (16, (1, 1, 1), 1, None)])
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "split_tf32", "split_f16", "split_bf16"])
def test_selfenergy_blocks(nao, kmesh, ntau, qr, sym, precision):
    # one X for (k, q, tau) and its image where P~ is symmetric, every block where it is not;
    # nao with and without whole 4 x 4 column blocks, odd and even tau counts
    naux = 19
    sysd = system(nao, naux, kmesh, ntau, 20.0, 91)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 92)
    P = hermitian_noise((km.nk, ntau, naux, naux), 0.3, 93)
    if sym:
        P = _folded(P, km)
    qs = list(range(km.nk) if qr is None else range(*qr))
    ref = ogw.selfenergy_tau(sysd["V"], G, P, km, qs=qs)
    g = gpu(sysd, precision=precision)
    if qr is not None:
        g.set_q_range(*qr)
    g.set("G_tau", G)
    g.set("P_tau", P)
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau"), ref) < TOL[precision]


@pytest.mark.parametrize("nao", [1, 2, 4, 7, 8, 9, 12, 15, 16, 17, 20])
@pytest.mark.parametrize("kmesh,ntau,naux", [((3, 1, 1), 5, 37), ((2, 1, 1), 3, 1), ((3, 2, 1), 2, 16)])
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("precision", ["split_f16", "split_bf16"])
def test_selfenergy_of_few_orbitals(nao, kmesh, ntau, naux, sym, precision):
    # the last two steps in one kernel up to nao 16 (one or two auxiliary functions per warp), GEMMs above
    sysd = system(nao, naux, kmesh, ntau, 20.0, 97)
    km = ogw.KMesh(kmesh)
    G = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 98)
    P = hermitian_noise((km.nk, ntau, naux, naux), 0.3, 99)
    if sym:
        P = _folded(P, km)
    ref = ogw.selfenergy_tau(sysd["V"], G, P, km, qs=list(range(km.nk)))
    g = gpu(sysd, precision=precision)
    g.set("G_tau", G)
    g.set("P_tau", P)
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau"), ref) < TOL[precision]


@pytest.mark.parametrize("kmesh,ntau", [((2, 1, 1), 5), ((3, 1, 1), 4)])
def test_polarization_vjp_blocks(kmesh, ntau):
    # the adjoint of the folded P~0 against the oracle's, which runs over every block
    from oracle import adjoint as oad
    import torch
    sysd = system(4, 11, kmesh, ntau, 20.0, 95)
    km = ogw.KMesh(kmesh)
    rng = np.random.default_rng(96)
    G = rng.standard_normal((ntau, km.nk, 4, 4)) + 1j * rng.standard_normal((ntau, km.nk, 4, 4))
    Pbar = rng.standard_normal((km.nk, ntau, 11, 11)) + 1j * rng.standard_normal((km.nk, ntau, 11, 11))
    g = gpu(sysd)
    g.set("G_tau", G)
    got = g.polarization_vjp(torch.from_numpy(Pbar).cuda()).cpu().numpy()
    assert rel(got, oad.polarization_vjp(sysd["V"], G, km, Pbar)) < 1e-12
