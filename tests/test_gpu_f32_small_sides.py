"""The FP32 operator on sides of 4 and 8 intervals, whose lines of 16 and 32
points are the shortest of the group transforms: both orders with every other
size of line, fewer rows than a block of pass A holds, one and several vectors,
truncated mode sets, and the allocation-free entry point, whose fixed scratch
is the workspace to the byte.  Reference: the FP64 operator on the same
vectors.  The pass options choose nothing: the same bits for every value.

Tolerance as for the larger sides (test_gpu_f32_operator.py): 1e-6, from at most
2 * 6 * 12 radix-2 stages of 2^-24 roundings in quadrature."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SIZES = [(4, 4), (4, 8), (8, 4), (8, 8), (4, 16), (16, 4), (8, 16), (16, 8), (32, 4), (4, 32),
         (8, 128), (128, 8), (256, 4), (4, 256), (512, 8), (8, 512), (1024, 4), (4, 1024)]


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2008_01966_gb300 as gb
    assert torch.cuda.is_available()
    return gb


def vectors(g, n, seed):
    rng = np.random.default_rng(seed)
    return torch.tensor(rng.standard_normal((n, g.n_ap)) + 1j * rng.standard_normal((n, g.n_ap)),
                        dtype=torch.complex64, device="cuda")


@pytest.mark.parametrize("nx, ny", SIZES)
@pytest.mark.parametrize("ndir, modes", [(1, 0), (5, 0), (2, 3)])
def test_small_sides_match_fp64(gb, nx, ny, ndir, modes):
    g = gb.Cavity(1.0, 1.0 if nx == ny else 0.75, 0.5, nx, ny, 8, precision="mixed", modes_m=modes,
                  modes_n=modes)
    g.prepare(2 * np.pi * min(nx, ny) / 10, [(4, 2.0 + 0.5j), (4, 1.0 + 0j)])
    x = vectors(g, ndir, nx + 7 * ny + ndir)
    ref = g.apply(x.to(torch.complex128), "fp64")
    y = g.apply(x, "mixed")
    for d in range(ndir):
        err = float(torch.linalg.vector_norm(y[d].to(torch.complex128) - ref[d]) /
                    torch.linalg.vector_norm(ref[d]))
        assert err < 1e-6, (d, err)
    try:
        z = g.apply_noalloc(x, "mixed")
    except gb.CavityError as e:
        assert e.status == 1      # more than the fixed scratch
    else:
        assert torch.equal(y, z)


@pytest.mark.parametrize("nx, ny", [(512, 512), (512, 64), (64, 512)])
def test_pass_options_choose_nothing(gb, nx, ny):
    g = gb.Cavity(1.0, 1.0 if nx == ny else 0.75, 0.5, nx, ny, 8, precision="mixed")
    g.prepare(2 * np.pi * min(nx, ny) / 10, [(4, 2.0 + 0.5j), (4, 1.0 + 0j)])
    x = vectors(g, 2, nx + ny)
    y = g.apply(x, "mixed")
    for b in (0, 1):
        for c in (0, 1):
            g.set_option("pass_b_2048", b)
            g.set_option("pass_c_2048", c)
            assert g.get_option("pass_b_2048") == b and g.get_option("pass_c_2048") == c
            assert torch.equal(g.apply(x, "mixed"), y), (b, c)
