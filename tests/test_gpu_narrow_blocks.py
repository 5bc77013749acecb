"""Mixed solves of one to nine directions: block Krylov bases of one to four
columns take kernels of their own for projection and update, five to eight
columns for the update, with half the tensor-core tile for the projection, nine
the whole tile; on grids smaller than a block's rows and on grids of several
slabs, and with repeated directions (dependent columns).

Check: the residual of the returned aperture under the FP64 operator.  The
solver stops at 1e-10 on its own residual, whose FP32 updates are within 1e-10
of it (see gmres.cu): 3e-10."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LAYERS = [(3, 4 + 1j), (3, 2 + 0.5j)]


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


@pytest.mark.parametrize("ndir", [1, 2, 3, 4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("same", [False, True])
@pytest.mark.parametrize("nx,ny", [(8, 8), (16, 32), (64, 64), (256, 128)])
def test_residual_of_narrow_batches(gb, nx, ny, ndir, same):
    g = gb.Cavity(1.0, 1.0 if nx == ny else 0.75, 0.25, nx, ny, 6, precision="mixed", gmres_tol=1e-10)
    th, ph, al = 0.2 + 0.15 * np.arange(ndir), 0.4 + 1.1 * np.arange(ndir), 0.3 * np.arange(ndir)
    if same:
        th[:], ph[:], al[:] = th[0], ph[0], al[0]
    x, _, it, res = g.solve(2 * np.pi * min(nx, ny) / 25, LAYERS, th, ph, al, field=False)
    assert np.all(res <= 1e-10), res
    rhs = g.rhs(th, ph, al)
    r = torch.linalg.vector_norm(rhs - g.apply(x, "fp64"), dim=1) / torch.linalg.vector_norm(rhs, dim=1)
    assert float(r.max()) <= 3e-10, r
