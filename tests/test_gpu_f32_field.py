"""The complex64 field at the sizes where its kernels change: the smallest and
largest lines, 4 to 64 lanes per line, both orders of a rectangle, sides of 8
intervals (which take the generic passes), with and without interfaces, one
and several directions, the smallest depth.  Reference: the FP64 field of the
same aperture vectors.

Tolerance: coefficients rounded once, then two lines of at most 11 radix-2
stages: about 2^-24 (1 + sqrt(2 * 11)) < 4e-7 for random coefficients; 1e-6 of
each level."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


@pytest.mark.parametrize("nx,ny", [(16, 16), (16, 32), (32, 16), (64, 64), (128, 32), (32, 256),
                                   (512, 16), (16, 512), (1024, 16), (16, 1024), (8, 32), (32, 8)])
@pytest.mark.parametrize("layers,ndir", [([(2, 2.0 + 0.5j)], 1), ([(5, 1.0 + 0j)], 3),
                                         ([(3, 4 + 1j), (2, 2 + 0.5j), (4, 1.0 + 0j)], 2)])
def test_field_matches_fp64(gb, nx, ny, layers, ndir):
    nz = sum(l for l, _ in layers)
    b = 1.0 if nx == ny else 0.75
    kap = 2 * np.pi * min(nx, ny) / 10
    out = {}
    for prec in ("fp64", "mixed"):
        g = gb.Cavity(1.0, b, 0.05, nx, ny, nz, precision=prec)
        g.prepare(kap, layers)
        rng = np.random.default_rng(nx + 5 * ny + ndir)
        x = torch.tensor(rng.standard_normal((ndir, g.n_ap)) + 1j * rng.standard_normal((ndir, g.n_ap)),
                         dtype=torch.complex128, device="cuda")
        out[prec] = g.field(x).to(torch.complex128).reshape(ndir, nz, -1)
    err = torch.linalg.vector_norm(out["mixed"] - out["fp64"], dim=2) / \
        torch.linalg.vector_norm(out["fp64"], dim=2)
    assert float(err.max()) < 1e-6, err
