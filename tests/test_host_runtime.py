"""The library's host side against a CUDA runtime without a GPU
(tests/fake_cuda.cpp): what it allocates, launches and sets up."""

import pytest

import fake_cuda


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


@pytest.fixture(autouse=True)
def fresh(fake):
    fake.lib.fake_reset()


def use(ctx):
    """The launches of one call of every operator and of the field."""
    n = ctx.lib.fake_log_size()
    assert [ctx.apply(2, p) for p in (0, 1, 2)] == [0, 0, 0] and ctx.field(2) == 0
    return [e for e in ctx.fake.log(n) if e.startswith("launch")]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_prepare_after_a_failed_allocation(fake, precision):
    """Whatever allocation of a prepare fails, the call reports it, the next
    prepare with the same arguments makes every table, and the kernels that
    follow get the pointers they get without the failure."""
    ctx = fake.context(precision=precision)
    fake.lib.fake_fail_alloc(0)
    n0 = fake.lib.fake_log_size()
    assert ctx.prepare(nlayers=2) == 0
    allocs = fake.lib.fake_allocs()
    made = {e for e in fake.log(n0) if e.startswith("launch")}
    want = use(ctx)
    ctx.close()
    for k in range(1, allocs + 1):
        ctx = fake.context(precision=precision)
        fake.lib.fake_fail_alloc(k)
        n0 = fake.lib.fake_log_size()
        assert ctx.prepare(nlayers=2) != 0
        assert b"memory" in fake.lib.cavity_last_error(ctx.h)
        fake.lib.fake_fail_alloc(0)
        assert ctx.prepare(nlayers=2) == 0, (k, fake.lib.cavity_last_error(ctx.h))
        assert made == {e for e in fake.log(n0) if e.startswith("launch")}, k   # by one or the other
        assert use(ctx) == want, k
        ctx.close()


def test_prepare_at_a_second_wavenumber_after_a_failure(fake):
    """A failure at a new wavenumber leaves no table of the old one in use."""
    ctx = fake.context()
    assert ctx.prepare(6.0) == 0
    fake.lib.fake_fail_alloc(1)
    assert ctx.prepare(7.0, nlayers=2) != 0     # the first allocation: the layered profiles
    fake.lib.fake_fail_alloc(0)
    n0 = fake.lib.fake_log_size()
    assert ctx.prepare(6.0) == 0
    assert any("k_khat(" in e for e in fake.log(n0))
    assert use(ctx)
    ctx.close()


def test_cross_section_of_many_directions(fake):
    """More directions than the second axis of a grid takes (65,535)."""
    ctx = fake.context(nx=16, ny=16)
    assert ctx.prepare() == 0
    assert ctx.rcs(65535) == 0 and ctx.rcs(70000) == 0
    ctx.close()


def test_field_of_many_slabs(fake):
    """Small grids with many directions and levels: more slabs than the third
    axis of a grid takes (65,535) go in several chunks."""
    ctx = fake.context(nx=16, ny=16, nz=8)
    assert ctx.prepare() == 0
    for ndir in (8192, 21000, 27500, 42000, 65535):
        assert ctx.field(ndir) == 0, ndir
    ctx.close()


@pytest.mark.parametrize("nx, ny, ndirs", [(16, 16, (1, 64, 300)), (32, 32, (8, 100, 256)),
                                           (64, 64, (1, 9, 64, 200, 600)), (64, 128, (17, 100)),
                                           (128, 128, (16, 64, 200)), (256, 256, (5, 16, 64)),
                                           (512, 512, (1, 8, 16))])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_footprint_is_an_upper_estimate(fake, nx, ny, ndirs, precision):
    """Serving admits contexts by footprint_bytes: what a context, its calls
    and their outputs allocate stays below it."""
    from paper_2008_01966_gb300.serving import footprint_bytes
    for ndir in ndirs:
        for nlayers in (1, 3):
            for field in (False, True):
                fake.lib.fake_reset()
                base = fake.lib.fake_live()
                ctx = fake.context(nx=nx, ny=ny, nz=12, precision=precision)
                assert ctx.solve(ndir, field=field, nlayers=nlayers) == 0 and ctx.rcs(ndir) == 0
                used = fake.lib.fake_peak() - base + ndir * ctx.n_ap * 16
                used += ndir * ctx.field_per_dir * ctx.el if field else 0
                ctx.close()
                assert used <= footprint_bytes((1.0, 1.0, 0.5, nx, ny, 12), ndir, precision,
                                               nlayers > 1, field), (ndir, nlayers, field)


def test_basis_of_a_group_is_as_wide_as_the_group(fake):
    """The block basis takes (steps + 1) x width columns per group."""
    def peak(width):
        fake.lib.fake_reset()
        base = fake.lib.fake_live()
        ctx = fake.context(nx=128, ny=128)
        assert fake.lib.cavity_set_option(ctx.h, 2, width) == 0
        assert ctx.solve(32, field=False) == 0
        used = fake.lib.fake_peak() - base
        n_ap = ctx.n_ap
        ctx.close()
        return used, n_ap

    (a, n_ap), (b, _) = peak(16), peak(4)
    # the same columns in all; what differs are the coefficients of more systems
    assert b - a < 0.05 * 31 * 32 * n_ap * 8


def test_every_device_is_set_up(fake):
    """Kernel attributes and constant tables belong to a device: the same calls
    on two devices set up the same on both."""
    def calls(dev):
        fake.lib.fake_set_device(dev)
        n = fake.lib.fake_log_size()
        for nx, solver, modes in ((8, "krylov", 0), (64, "krylov", 0), (32, "dense", 6)):
            for precision in ("fp64", "mixed"):
                ctx = fake.context(nx=nx, ny=nx, precision=precision, solver=solver, modes=modes)
                ctx.prepare()
                use(ctx)
                ctx.solve(20)
                ctx.close()
        return sorted(e.replace("device=%d" % dev, "") for e in fake.log(n)
                      if e.startswith(("symbol", "attribute")) and e.endswith("device=%d" % dev))

    first, second = calls(11), calls(12)
    assert any("g_j0_tab" in e for e in first) and any("k_opB" in e for e in first)
    assert any("k_lu_panel_cluster" in e for e in first)
    assert first == second


def test_lu_factor_after_lu_solve(fake):
    """A solve with given factors, as the first dense call on a device, leaves
    the factorisation's kernel its own setting."""
    import ctypes
    import numpy as np
    fake.lib.fake_set_device(21)
    ctx = fake.context()
    assert ctx.prepare() == 0
    n = 4000
    a, b = np.empty(n * n * 2, np.float32), np.empty(n * 2, np.float32)
    piv = np.zeros(n, np.int32)
    p = lambda v: ctypes.c_void_p(v.ctypes.data)  # noqa: E731
    start = fake.lib.fake_log_size()
    assert ctx.lib.cavity_lu_solve(ctx.h, p(a), 64, 64, p(piv), 1, p(b), 64) == 0
    ctx.lib.cavity_lu_factor(ctx.h, p(a), n, n, p(piv), None)
    log = fake.log(start)
    assert any(e.startswith("launch k_lu_panel(") for e in log)
    assert any(e.startswith("attribute") and "k_lu_panel(" in e for e in log)
    ctx.close()


@pytest.mark.parametrize("nx, nz, ndir, chunks", [(512, 16, 1, 8), (512, 9, 2, 5), (512, 64, 8, 8),
                                                  (256, 64, 1, 8), (64, 32, 1, 1), (64, 32, 64, 1),
                                                  (16, 8, 1, 1)])
def test_host_field_leaves_in_chunks(fake, nx, nz, ndir, chunks):
    """A field for the host is synthesised and copied in several chunks, so
    that the copy overlaps the synthesis; small ones in one, whose copies are not
    worth splitting."""
    ctx = fake.context(nx=nx, ny=nx, nz=nz)
    assert ctx.prepare() == 0
    n = fake.lib.fake_log_size()
    assert ctx.solve(ndir, host=True) == 0
    assert sum("k_fy<" in e and e.startswith("launch") for e in fake.log(n)) == chunks
    level = ctx.field_per_dir // nz * 8
    sizes = [int(e.split()[1]) for e in fake.log(n) if e.startswith("download")]
    assert sum(s for s in sizes if s % level == 0) == ndir * nz * level   # every level once
    ctx.close()


def test_no_launch_overtakes_a_copy_on_the_default_stream(fake):
    """A context's stream may be one that does not wait for the default stream:
    what is copied there has to be waited for before anything is launched."""
    fake.lib.fake_set_device(31)
    for solver, modes in (("krylov", 0), ("dense", 6)):
        ctx = fake.context(stream=0x1000, solver=solver, modes=modes)
        n = fake.lib.fake_log_size()
        ctx.prepare()
        pending = None
        for e in fake.log(n):
            if e.startswith("copy on the default") or (e.startswith("symbol") and " async" not in e):
                pending = e
            elif e == "sync default":
                pending = None
            assert not (pending and e.startswith("launch")), (pending, e)
        ctx.close()
