"""LU panels on a cluster of blocks: sizes around the rows per block and the
panel width, and one whose first panels are too tall for the cluster, so that
both panel kernels run in one factorisation.

Check: P A = L U within the bound of the partial-pivoting test (2e-6 sqrt(n)
of the largest entry), multipliers of at most 1, every step exchanging rows."""

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


@pytest.mark.parametrize("n", [2, 15, 17, 63, 66, 95, 97, 129, 577, 1024, 2081, 3200])
def test_factors_reproduce_the_matrix(gb, n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    a = torch.view_as_complex(torch.randn((n, n, 2), generator=gen, device="cuda"))
    a.fill_diagonal_(0)
    full = a.to(torch.complex128)
    g = gb.Cavity(1.0, 1.0, 0.5, 8, 8, 4)
    ipiv, info = g.lu_factor(a)
    assert info == -1
    piv = ipiv.cpu().numpy()
    assert np.all((piv >= np.arange(n)) & (piv < n))
    perm = np.arange(n)
    for i, p in enumerate(piv):
        perm[[i, p]] = perm[[p, i]]
    lu = a.to(torch.complex128)
    low = torch.tril(lu, -1)
    assert float(low.abs().max()) <= 1 + 1e-6
    low.diagonal().fill_(1)
    err = float((low @ torch.triu(lu) - full[torch.from_numpy(perm).cuda()]).abs().max() / full.abs().max())
    assert err < 2e-6 * np.sqrt(n), err
