"""Device memory of a 2D handle: the vectors that only a multigrid preconditioner reads are allocated only
with one.  1024^2 cells, 20 pairs, restart length 1, in cell arrays of 8 bytes: 11 x 20 pair arrays
(E, O, the diagonals, vertex values, right-hand side parts and work), 2 x 2 rho rows, 2 basis
vectors of 21 and about 20 cell arrays, 286 together; mixed precision adds 2 x 21/2 + 20 + 4.
Another 2 x 21 (and 21/2) would be the multigrid vectors.  Allowed above the count: 10 arrays and 64
MB for the allocator's rounding."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed,arrays", [(False, 286), (True, 331)])
def test_no_multigrid_vectors_by_default(mixed, arrays):
    import torch
    from paper_1811_05579_gb300 import grte as G

    def used(n, prec):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        h = G.Grte2D(n, n, 1.0, 1e-3, 1e-1, krylov_restart=1, precision=G.MIXED if mixed else G.FP64, prec=prec)
        torch.cuda.synchronize()
        took = free - torch.cuda.mem_get_info()[0]
        h.close()
        return took

    used(16, 0)     # what the library loads with its first handle
    n = 1024
    assert used(n, 0) <= (arrays + 10) * 8 * n * n + (64 << 20)
