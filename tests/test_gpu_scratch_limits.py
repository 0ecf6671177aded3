"""A context of the 16-bit chains on an allocator without room for the workspaces that only save launches and
traffic: it is created, and its results are those of one with room, also after values that are not finite have
been through the memory that the two chains then share."""
import numpy as np
import pytest

from gpu_helpers import gpu, hermitian_noise, rel, system
from oracle import gw as ogw

pytestmark = pytest.mark.gpu


class Allocator:
    """PyTorch's allocator with a limit on the bytes in use (None: no limit), or without room for one size."""

    def __init__(self, monkeypatch):
        import torch
        self.limit, self.refused, self.live = None, None, {}
        alloc, free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete

        def take(n, *where):
            if n == self.refused:
                raise RuntimeError("size")
            if self.limit is not None and sum(self.live.values()) + n > self.limit:
                raise RuntimeError("limit")
            p = alloc(n, *where)
            self.live[p] = n
            return p

        def give(p):
            self.live.pop(p)
            free(p)
        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", take)
        monkeypatch.setattr(torch.cuda, "caching_allocator_delete", give)


@pytest.mark.parametrize("nao,naux,kmesh,ntau", [(18, 33, (3, 1, 1), 9), (8, 20, (2, 2, 1), 10), (5, 17, (3, 1, 1), 7),
                                                 (32, 21, (2, 1, 1), 6)])
@pytest.mark.parametrize("precision,tol", [("split_f16", 5e-6), ("split_bf16", 5e-5)])
def test_without_room_for_the_pieces_of_x(monkeypatch, nao, naux, kmesh, ntau, precision, tol):
    import torch
    torch.cuda.set_device(0)
    mem = Allocator(monkeypatch)
    sysd = system(nao, naux, kmesh, ntau, 20.0, 171)
    km = ogw.KMesh(kmesh)
    G, P = hermitian_noise((ntau, km.nk, nao, nao), 0.3, 172), hermitian_noise((km.nk, ntau, naux, naux), 0.3, 173)
    full = gpu(sysd, precision=precision)
    sizes = sorted(mem.live.values())
    one = ntau * 2 * ((2 * nao + 15) // 16) * naux * nao * 16       # one plane of X's pieces of one k
    planes = [s for s in sizes if s > 2048 and (s - 2048) % one == 0 and sizes.count(s) >= 4]
    assert planes
    if nao == 32:   # (the shared memory has the planes' size there)
        mem.limit = sum(sizes) - 4 * planes[0] + 4 * 2048 + 65536
    else:
        mem.refused = planes[0]
    full.close()
    assert not mem.live
    g = gpu(sysd, precision=precision)
    for bad in (True, False, False):
        g.set("G_tau", G + (np.inf if bad else 0.0))
        g.set("P_tau", P + (np.inf if bad else 0.0))
        g.selfenergy_partial()
        g.polarization()
    assert rel(g.get("P0_tau"), ogw.polarization_tau(sysd["V"], G, km)) < tol
    g.set("P_tau", P)
    g.selfenergy_partial()
    assert rel(g.get("Sigma_tau"), ogw.selfenergy_tau(sysd["V"], G, P, km, qs=list(range(km.nk)))) < tol
