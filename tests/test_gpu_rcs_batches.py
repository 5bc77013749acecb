"""Cross-sections of one direction, a few and many: the same bits (the sums are
formed in an order that depends on the grid alone), and the values of a plain
sum in 64 bits.

Tolerance against the plain sum: 3 nx ny terms of one sign at worst, each with
a few roundings, in another order: 1e-13 of sum |term| squared, generously."""

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


def integrals(kind, n, side, g):
    def ef(s):
        return side * np.exp(-0.5j * s * side) * np.sinc(0.5 * s * side / np.pi)
    k = np.arange(n) * np.pi / side
    return 0.5 * (ef(g - k) + ef(g + k)) if kind == "c" else (ef(g - k) - ef(g + k)) / 2j


@pytest.mark.parametrize("nx, ny, many", [(4, 4, 1500), (8, 4, 700), (4, 64, 300), (16, 16, 5000),
                                          (16, 32, 500), (64, 16, 600), (64, 64, 700),
                                          (1024, 4, 300), (4, 1024, 300), (128, 64, 90),
                                          (512, 256, 40)])
def test_sums(gb, nx, ny, many):
    b = {True: 1.0, False: 0.75 if ny < nx else 1.5}[nx == ny]
    g = gb.Cavity(1.0, b, 0.5, nx, ny, 4, precision="mixed")
    kappa0 = 7.3
    g.prepare(kappa0, [(4, 1.0 + 0j)])
    rng = np.random.default_rng(nx + 7 * ny)
    ap = torch.tensor(rng.standard_normal((many, g.n_ap)) + 1j * rng.standard_normal((many, g.n_ap)),
                      dtype=torch.complex128, device="cuda")
    th, ph = rng.uniform(0, 1.2, many), rng.uniform(0, 6.2, many)
    for pol in ("theta", "phi"):
        sig = g.rcs(ap, th, ph, pol)
        for d in (0, 1, many // 2, many - 1):
            assert g.rcs(ap[d:d + 1], th[d:d + 1], ph[d:d + 1], pol)[0] == sig[d], d
            x = ap[d].cpu().numpy()
            E1 = x[:g.n1].reshape(nx, ny - 1)
            E2 = x[g.n1:g.n1 + g.n2].reshape(nx - 1, ny)
            t, f = th[d], ph[d]
            xh = np.array([np.sin(t) * np.cos(f), np.sin(t) * np.sin(f), np.cos(t)])
            e = np.array([np.cos(t) * np.cos(f), np.cos(t) * np.sin(f), -np.sin(t)]) \
                if pol == "theta" else np.array([-np.sin(f), np.cos(f), 0.0])
            c1, s2 = (integrals(k, nx, 1.0, kappa0 * xh[0]) for k in "cs")
            s1, c2 = (integrals(k, ny, b, kappa0 * xh[1]) for k in "sc")
            terms1, terms2 = c1[:, None] * E1 * s1[None, 1:], s2[1:, None] * E2 * c2[None, :]
            L = np.array([-terms2.sum(), terms1.sum(), 0.0])
            want = kappa0 ** 2 / np.pi * abs(np.dot(e, np.cross(xh, L))) ** 2
            scale = kappa0 ** 2 / np.pi * (np.abs(terms1).sum() + np.abs(terms2).sum()) ** 2
            assert abs(sig[d] - want) <= 1e-13 * scale, (d, pol)
