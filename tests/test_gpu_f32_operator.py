"""The FP32 operator at the sizes where its dispatch and its group transforms
change: the smallest and largest sides, every number of lanes per line (8 to
128), both orders of a rectangle, sides of 8 intervals (which take the generic
passes), one and several vectors, a truncated mode set.  Reference: the FP64
operator on the same vectors.

Tolerance: a line passes six transforms of at most 12 radix-2 stages per axis
pair, so the relative error is about 2^-24 sqrt(2 * 6 * 12) * 1/2 < 4e-7 for
random vectors; 1e-6."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SIZES = [(16, 16), (16, 32), (32, 16), (64, 64), (128, 32), (32, 256), (256, 128), (512, 16),
         (16, 512), (1024, 16), (16, 1024), (8, 64), (64, 8), (1024, 512)]


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("ndir,modes", [(1, 0), (3, 0), (2, 5)])
def test_fp32_operator_matches_fp64(gb, nx, ny, ndir, modes):
    b = 1.0 if nx == ny else 0.75
    g = gb.Cavity(1.0, b, 0.5, nx, ny, 8, precision="mixed", modes_m=modes, modes_n=modes)
    g.prepare(2 * np.pi * min(nx, ny) / 10, [(4, 2.0 + 0.5j), (4, 1.0 + 0j)])
    rng = np.random.default_rng(nx + 7 * ny + ndir)
    x = torch.tensor(rng.standard_normal((ndir, g.n_ap)) + 1j * rng.standard_normal((ndir, g.n_ap)),
                     dtype=torch.complex64, device="cuda")
    ref = g.apply(x.to(torch.complex128), "fp64")
    y = g.apply(x, "mixed").to(torch.complex128)
    for d in range(ndir):
        err = float(torch.linalg.vector_norm(y[d] - ref[d]) / torch.linalg.vector_norm(ref[d]))
        assert err < 1e-6, (d, err)
