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
