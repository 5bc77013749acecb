"""A vector's FP64 and pair-of-FP32 results do not depend on the batch: the
operator on one vector, on a few and on many takes different launches (lines
per block, pass B of one column per block for small launches), which give the
same bits, and so does an FP64 solve, whose sums are formed in a fixed order
that depends on the grid alone."""

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


SIZES = [(4, 4), (8, 16), (16, 8), (16, 64), (64, 16), (32, 32), (64, 64), (128, 64), (128, 128),
         (256, 32)]


@pytest.mark.parametrize("precision", ["fp64", "pair32"])
@pytest.mark.parametrize("nx, ny", SIZES)
def test_operator_bits(gb, nx, ny, precision):
    g = gb.Cavity(1.0, 1.0 if nx == ny else 0.75, 0.5, nx, ny, 6, precision="mixed")
    g.prepare(2 * np.pi * min(nx, ny) / 10, [(3, 2.0 + 0.5j), (3, 1.0 + 0j)])
    rng = np.random.default_rng(nx + 3 * ny)
    x = torch.tensor(rng.standard_normal((48, g.n_ap)) + 1j * rng.standard_normal((48, g.n_ap)),
                     dtype=torch.complex128, device="cuda")
    y = g.apply(x, precision)
    for n in (1, 2, 3, 5, 9, 20):
        assert torch.equal(g.apply(x[:n].contiguous(), precision), y[:n]), n


@pytest.mark.parametrize("nx, ny", [(8, 8), (16, 16), (64, 16), (32, 32), (64, 64)])
def test_fp64_solve_bits(gb, nx, ny):
    g = gb.Cavity(1.0, 1.0 if nx == ny else 0.75, 0.5, nx, ny, 6, precision="fp64")
    layers, kappa0 = [(3, 2.0 + 0.5j), (3, 1.0 + 0j)], 2 * np.pi * min(nx, ny) / 10
    rng = np.random.default_rng(nx)
    th, ph, al = rng.uniform(0, 1, 24), rng.uniform(0, 6, 24), rng.uniform(0, 1, 24)
    ap, fl, _, _ = g.solve(kappa0, layers, th, ph, al)
    for n in (1, 3, 8):
        a, f, _, _ = g.solve(kappa0, layers, th[:n], ph[:n], al[:n])
        assert torch.equal(a, ap[:n]) and torch.equal(f, fl[:n]), n
