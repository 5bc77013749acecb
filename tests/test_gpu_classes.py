"""Mixed solves on grids large enough for the parity classes of the block
Krylov solver (300,000 unknowns and more): batches whose classes are empty
(normal incidence), one-dimensional (directions in a mirror plane), dependent
(repeated directions) or all of these at once, on a square and on rectangles,
with a truncated mode set, restarts of the basis, and one direction alone.

Check: the residual of the returned aperture under the FP64 operator.  The
solver stops at 1e-10 on its own residual, whose FP32 updates are within 1e-10
of it (see gmres.cu): 3e-10."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LAYERS = [(3, 4 + 1j), (3, 2 + 0.5j)]
ZERO = (0.0, 0.0, 0.0)
PLANE = (0.6, 0.0, 0.0)
ANY = (0.9, 0.7, 0.3)
OTHER = (0.4, 4.1, 1.2)


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


@pytest.mark.parametrize("dirs", [[ZERO], [ANY], [PLANE, PLANE], [ZERO, ANY, ANY, PLANE, OTHER],
                                  [ANY, OTHER] * 9])
@pytest.mark.parametrize("nx,ny,b,kw", [(512, 512, 1.0, {}), (512, 256, 0.75, {}),
                                        (256, 512, 1.5, dict(modes_m=100, modes_n=60)),
                                        (512, 256, 0.5, dict(gmres_restart=4))])
def test_residual_of_degenerate_batches(gb, nx, ny, b, kw, dirs):
    g = gb.Cavity(1.0, b, 0.25, nx, ny, 6, precision="mixed", gmres_tol=1e-10, **kw)
    th, ph, al = (np.array(v) for v in zip(*dirs))
    x, _, it, res = g.solve(40.0, LAYERS, th, ph, al, field=False)
    assert np.all(res <= 1e-10), res
    rhs = g.rhs(th, ph, al)
    if kw.get("modes_m"):
        # the rows of the dropped modes are zero in A x; drop them from b as well
        mask = (g.apply(torch.ones_like(rhs[:1]), "fp64")[0] != 0).to(rhs.dtype)
        rhs = rhs * mask
    r = torch.linalg.vector_norm(rhs - g.apply(x, "fp64"), dim=1) / torch.linalg.vector_norm(rhs, dim=1)
    assert float(r.max()) <= 3e-10, r
