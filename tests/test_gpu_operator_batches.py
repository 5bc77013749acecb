"""FP64 and pair-of-FP32 operators: a vector alone and the same vector in a
batch.  The launches differ (lines per block, and pass B of one column per
block for small launches), the arithmetic does not beyond the order of sums.

Tolerance: a value takes about 100 roundings either way (a few transforms of
up to 10 stages), in another order: 2 * 10 units of 2^-53 and, in pair
arithmetic, of 2^-46 at most: 1e-14 (rounded up) and 1e-12."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-14, "pair32": 1e-12}


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


@pytest.mark.parametrize("precision", ["fp64", "pair32"])
@pytest.mark.parametrize("nx,ny,batch", [(4, 4, 200), (8, 16, 60), (16, 8, 80), (32, 32, 24),
                                         (128, 64, 12), (64, 128, 6), (128, 128, 8), (256, 32, 24)])
def test_alone_and_in_a_batch(gb, nx, ny, batch, precision):
    g = gb.Cavity(1.0, 1.0 if nx == ny else 0.75, 0.5, nx, ny, 6, precision="mixed")
    g.prepare(2 * np.pi * min(nx, ny) / 10, [(3, 2.0 + 0.5j), (3, 1.0 + 0j)])
    rng = np.random.default_rng(nx + 3 * ny)
    x = torch.tensor(rng.standard_normal((batch, g.n_ap)) + 1j * rng.standard_normal((batch, g.n_ap)),
                     dtype=torch.complex128, device="cuda")
    y = g.apply(x, precision)
    for d in (0, batch - 1):
        one = g.apply(x[d:d + 1], precision)[0]
        err = float(torch.linalg.vector_norm(one - y[d]) / torch.linalg.vector_norm(y[d]))
        assert err < TOL[precision], (d, err)
