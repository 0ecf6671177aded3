"""P~0 folded over (q, tau) -> (-q, beta - tau): only half of the (q, tau) blocks are
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
