"""Tables of a wavenumber at the edges of their evaluation: the kernel table on
square and unequal periods (the symmetric half is evaluated once) across the
switches of J0 (argument 25) and of the large-argument form; right-hand sides
whose trapezoid progressions have a ratio at or next to 1.  Reference: the
oracle, which sums both term by term.

Tolerances.  Table: the oracle's quadrature loses about c R 1e-16 relative to
the rounding of its arguments, c R < 400 here: 1e-12 per entry with 1e-15 of
the largest.  Right-hand side: sums of 17 unit terms, whose angles round to
1e-15 relative at most 30 pi: 1e-12 of the largest entry."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.excitation import rhs
from oracle.geometry import Cavity as OCavity, Layer
from oracle.khat import khat

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


@pytest.mark.parametrize("nx,ny,b", [(16, 16, 1.0), (32, 16, 1.0), (16, 32, 1.0), (16, 16, 0.75),
                                     (32, 16, 0.5), (64, 64, 1.0)])
@pytest.mark.parametrize("kappa0", [0.3, 17.6, 40.0])
def test_kernel_table(gb, nx, ny, b, kappa0):
    g = gb.Cavity(1.0, b, 0.5, nx, ny, 4)
    g.prepare(kappa0, [(4, 2.0 + 0.5j)])
    t = g.export_khat().cpu().numpy()
    j1, j2 = np.arange(t.shape[0]), np.arange(t.shape[1])
    rho = np.hypot(j1[:, None] / 4.0, j2[None, :] / (4.0 * b))
    ref = khat(rho, kappa0, np.sqrt(2.0))
    err = np.abs(t - ref)
    assert np.all(err <= 1e-12 * np.abs(ref) + 1e-15 * np.abs(ref).max()), err.max()
    if b == 1.0:
        k = min(nx, ny) * 2
        assert np.array_equal(t[:k, :k], t[:k, :k].T)


@pytest.mark.parametrize("delta", [0.0, 1e-13, 1e-9, 1e-5, 1e-2, 3.1e-2, 3.3e-2])
@pytest.mark.parametrize("nx,ny,m", [(16, 16, 3), (16, 32, 0), (32, 16, 9)])
def test_rhs_progressions(gb, nx, ny, m, delta):
    kap = np.pi * m + delta + 1e-3 * (m == 0)
    g = gb.Cavity(1.0, 1.0, 0.5, nx, ny, 4)
    g.prepare(kap, [(4, 2.0 + 0.5j)])
    th, ph, al = np.full(4, np.pi / 2), np.array([0, np.pi / 2, np.pi, -np.pi / 2]), np.full(4, 0.4)
    out = g.rhs(th, ph, al).cpu().numpy()
    cav = OCavity(1.0, 1.0, 0.5, nx, ny, 4, kap, layers=[Layer(4, 2.0 + 0.5j)])
    for d in range(4):
        ref = rhs(cav, th[d], ph[d], al[d])
        assert np.abs(out[d] - ref).max() <= 1e-12 * np.abs(ref).max(), d
