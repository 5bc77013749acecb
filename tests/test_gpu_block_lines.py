"""FP64 and pair-of-FP32 operators on sides of 256 intervals and more, where the
threads of a block, the points per thread and the number of line groups of the
block transforms change (1024-, 2048- and 4096-point lines), with small and
large batches.  Each arithmetic is the other's reference.

Tolerance: a value takes about 100 roundings either way, of 2^-53 and of 2^-46
at most: 100 * 2^-46 = 1.4e-12 in the worst case of all of one sign; 1e-12."""

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


@pytest.mark.parametrize("nx,ny,ndir", [(256, 16, 1), (256, 64, 5), (512, 16, 1), (16, 512, 1),
                                        (512, 64, 5), (64, 512, 5), (1024, 16, 1), (16, 1024, 1),
                                        (1024, 512, 2), (512, 1024, 1)])
def test_pair_and_fp64_agree(gb, nx, ny, ndir):
    g = gb.Cavity(1.0, 0.75, 0.5, nx, ny, 6, precision="mixed")
    g.prepare(2 * np.pi * min(nx, ny) / 10, [(3, 2.0 + 0.5j), (3, 1.0 + 0j)])
    rng = np.random.default_rng(nx + 3 * ny)
    x = torch.tensor(rng.standard_normal((ndir, g.n_ap)) + 1j * rng.standard_normal((ndir, g.n_ap)),
                     dtype=torch.complex128, device="cuda")
    y, z = g.apply(x, "fp64"), g.apply(x, "pair32")
    for d in range(ndir):
        err = float(torch.linalg.vector_norm(y[d] - z[d]) / torch.linalg.vector_norm(y[d]))
        assert err < 1e-12, (d, err)
