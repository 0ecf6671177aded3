"""What the adjoints of a mixed-precision context allocate: the digit workspaces belong to the FP64 adjoints."""
import numpy as np
import pytest

from gpu_helpers import gpu, hermitian_noise, system
from oracle import gw as ogw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "split_f16"])
def test_complex64_adjoints_and_tangents_allocate_no_digits(precision):
    import torch
    nao, naux, kmesh, ntau = 13, 97, (2, 1, 1), 41    # above the size from which FP64 products take digits
    sysd = system(nao, naux, kmesh, ntau, 20.0, 131)
    nk, n2, na2 = ogw.KMesh(kmesh).nk, nao * nao, naux * naux
    g = gpu(sysd, precision=precision)
    g.set("G_tau", hermitian_noise((ntau, nk, nao, nao), 0.3, 132))
    P0 = hermitian_noise((nk, ntau, naux, naux), 0.01, 133)
    g.set("P0_iw", P0)
    g.screened()
    g.set("P_tau", hermitian_noise((nk, ntau, naux, naux), 0.3, 134))
    dev = [torch.from_numpy(x).cuda() for x in (P0, hermitian_noise((ntau, nk, nao, nao), 0.3, 135))]
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    for call in (lambda: g.polarization_vjp(dev[0], c64=True), lambda: g.selfenergy_vjp(dev[1], c64=True),
                 lambda: g.screened_jvp(dev[0])):
        call()
    torch.cuda.synchronize()
    # three chain buffers and the complex64 copies of G, P~ and one cotangent; 2 MB for the allocator's rounding
    buffers = 3 * 16 * max(ntau * naux * n2, ntau * na2, ntau * nk * n2)
    copies = 8 * (ntau * nk * n2 + nk * ntau * na2 + max(ntau * na2, ntau * nk * n2))
    assert torch.cuda.memory_allocated() - before <= buffers + copies + (2 << 20)
    # the FP64 adjoint has them, and its result is the complex64 one's to single precision
    a, b = (g.polarization_vjp(dev[0], c64=c).cpu().numpy() for c in (False, True))
    assert torch.cuda.memory_allocated() - before > buffers + copies + (2 << 20)
    assert np.abs(a - b).max() < 1e-5 * np.abs(a).max()
