"""The symmetries that the folded routes rest on are looked at before they are used: data without them,
or with a value that is not finite, take the route over every block."""
import numpy as np
import pytest

from gpu_helpers import gpu, hermitian_noise, system
from oracle import gw as ogw

pytestmark = pytest.mark.gpu

NAO, NAUX, KMESH, NTAU = 4, 18, (3, 1, 1), 14


def _context(**kw):
    return gpu(system(NAO, NAUX, KMESH, NTAU, 20.0, 121), **kw)


def _fails_or_not_finite(call, result):
    """An error of the library, or a result that shows the value."""
    from paper_2206_07660_gb300.gw import GWError
    try:
        call()
    except GWError:
        return True
    return not np.isfinite(result()).all()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("q,m", [(0, 0), (1, 0), (2, NTAU - 1), (0, NTAU - 1)])
def test_p0_iw_that_is_not_finite(value, q, m):
    # frequencies and q-points that the fold keeps, and ones that it takes from their partners
    sysd = system(NAO, NAUX, KMESH, NTAU, 20.0, 121)
    st = ogw.State(sysd)
    st.G_tau = -hermitian_noise((NTAU, 3, NAO, NAO), 0.05, 122) - 0.3 * np.eye(NAO)
    st.sigma()
    P0 = st.P0_iw.copy()
    P0[q, m, 2, 3] = value
    g = gpu(sysd)
    g.set("P0_iw", P0)
    assert _fails_or_not_finite(g.screened, lambda: g.get("P_iw")[q, m])


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("q,t", [(0, 0), (0, NTAU - 1), (2, 3)])
@pytest.mark.parametrize("precision", ["fp64", "split_f16"])
def test_p_tau_that_is_not_finite(value, q, t, precision):
    km = ogw.KMesh(KMESH)
    P = hermitian_noise((km.nk, NTAU, NAUX, NAUX), 0.3, 123)
    neg = [km.index(-km.vec[i]) for i in range(km.nk)]
    P = 0.5 * (P + np.conj(P[neg][:, ::-1]))
    P[q, t, 1, 1] = value
    g = _context(precision=precision)
    g.set("G_tau", hermitian_noise((NTAU, km.nk, NAO, NAO), 0.3, 124))
    g.set("P_tau", P)
    assert _fails_or_not_finite(g.selfenergy_partial, lambda: g.get("Sigma_tau")[t])


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("w", [0, NTAU - 1])
def test_sigma_iw_that_is_not_finite(value, w):
    g = _context()
    S = np.zeros(g.shape_of("Sigma_iw"), dtype=np.complex128)
    S[w, 1, 2, 2] = value
    g.set("Sigma_iw", S)
    assert _fails_or_not_finite(g.dyson, lambda: g.get("G_iw")[w])


@pytest.mark.parametrize("stage", ["forward", "tangent"])
def test_captured_selfenergy_is_replayed_on_other_p_tau(stage):
    # a stage captured after a symmetric P~ serves a P~ without the symmetry that is handed in later
    import torch
    km = ogw.KMesh(KMESH)
    sysd = system(NAO, NAUX, KMESH, NTAU, 20.0, 121)
    neg = [km.index(-km.vec[i]) for i in range(km.nk)]
    G = hermitian_noise((NTAU, km.nk, NAO, NAO), 0.3, 125)
    P = hermitian_noise((km.nk, NTAU, NAUX, NAUX), 0.3, 126)
    sym = 0.5 * (P + np.conj(P[neg][:, ::-1]))
    dG, dP = hermitian_noise(G.shape, 0.3, 127), hermitian_noise(P.shape, 0.3, 128)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        g = gpu(sysd)
        dGd, dPd = torch.from_numpy(dG).cuda(), torch.from_numpy(dP).cuda()
        out = {}

        def run():
            if stage == "forward":
                g.selfenergy_partial()
            else:
                out["S"] = g.selfenergy_jvp(dGd, dPd)

        g.set("G_tau", G)
        g.set("P_tau", sym)
        g.selfenergy_partial()
        run()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            run()
        g.set("P_tau", P)
        graph.replay()
        torch.cuda.synchronize()
        got = g.get("Sigma_tau") if stage == "forward" else out["S"].cpu().numpy()
    qs = list(range(km.nk))
    if stage == "forward":
        ref = ogw.selfenergy_tau(sysd["V"], G, P, km, qs=qs)
    else:
        ref = ogw.selfenergy_tau(sysd["V"], dG, P, km, qs=qs) + ogw.selfenergy_tau(sysd["V"], G, dP, km, qs=qs)
    assert np.abs(got - ref).max() < 1e-12 * np.abs(ref).max()


def test_capture_of_the_iteration_leaves_a_given_p_tau_unfolded():
    # the graph is captured without being run: the P~ that is in place is still the caller's
    km = ogw.KMesh(KMESH)
    sysd = system(NAO, NAUX, KMESH, 24, 20.0, 129)
    g = gpu(sysd)
    g.iterate(1)
    G = g.get("G_tau")
    P = hermitian_noise((km.nk, 24, NAUX, NAUX), 0.3, 130)
    g.set("P_tau", P)
    g.iterate_graph(0)
    g.selfenergy_partial()
    ref = ogw.selfenergy_tau(sysd["V"], G, P, km, qs=list(range(km.nk)))
    assert np.abs(g.get("Sigma_tau") - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("defect", [0.0, 5e-12])
def test_sigma_inf_of_loosely_paired_v(defect):
    # Sigma_inf is made Hermitian where V is paired; a pairing defect that the checks accept stays in it
    sysd = system(NAO, NAUX, KMESH, 24, 20.0, 136)
    rng = np.random.default_rng(137)
    V = sysd["V"] * (1.0 + defect * rng.standard_normal(sysd["V"].shape))
    st = ogw.State(sysd)
    G = -hermitian_noise((24, 3, NAO, NAO), 0.05, 138) - 0.3 * np.eye(NAO)
    gamma = ogw.density_matrix(st.grid, G)
    ref = ogw.hartree(V, gamma) + ogw.exchange(V, gamma)
    g = gpu(dict(sysd, V=V))
    g.set("G_tau", G)
    g.hf()
    got = g.get("Sigma_inf_new")
    assert np.abs(got - ref).max() < 2e-14 * np.abs(ref).max()
    if defect == 0.0:
        assert np.array_equal(got, np.conj(np.swapaxes(got, -1, -2)))


@pytest.mark.parametrize("matrix", ["TBb", "TFb", "TFf"])
def test_callers_grid_is_applied_as_given(matrix):
    # transforms that miss their mirror symmetry by more than rounding are not replaced by their symmetric part
    sysd = system(NAO, NAUX, KMESH, NTAU, 20.0, 139)
    st = ogw.State(sysd)
    grid = {k: np.array(getattr(st.grid, k)) for k in ("tau", "TFf", "TBf", "TFb", "TBb", "lb")}
    grid["fermi_n"], grid["bose_m"] = sysd["fermi_n"], sysd["bose_m"]
    rng = np.random.default_rng(140)
    defect = {"TBb": 4e-12, "TFb": 3e-14, "TFf": 3e-14}[matrix]
    grid[matrix] = grid[matrix] + defect * np.abs(grid[matrix]).max() * rng.uniform(-1, 1, grid[matrix].shape)
    import torch
    from paper_2206_07660_gb300 import GW
    torch.cuda.set_device(0)
    g = GW(sysd["H0"], sysd["S"], sysd["V"], KMESH, NTAU, 20.0, n_elec=sysd["n_elec"], grid=grid, damping=1.0)
    g.set("G_tau", -hermitian_noise((NTAU, 3, NAO, NAO), 0.05, 141) - 0.3 * np.eye(NAO))
    g.polarization()
    p0_tau, p0_iw = g.get("P0_tau"), g.get("P0_iw")
    g.screened()
    p_iw, p_tau = g.get("P_iw"), g.get("P_tau")
    g.selfenergy()
    for T, x, y, axis in ((grid["TFb"], p0_tau, p0_iw, 1), (grid["TBb"], p_iw, p_tau, 1),
                          (grid["TFf"], g.get("Sigma_tau"), g.get("Sigma_iw"), 0)):
        ref = ogw.to_matsubara(T, x, axis)
        if axis == 1 and T is grid["TBb"]:
            ref = ogw.herm(ref)
        # sums of 14 terms: a few units in the last place of the largest possible one
        assert np.abs(y - ref).max() < 1e-15 * np.abs(T).sum(1).max() * np.abs(x).max()
