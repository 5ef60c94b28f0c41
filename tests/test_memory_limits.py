"""What the library does when device memory is short, on the host: its objects
linked with a CUDA runtime whose device memory is host memory with a settable
capacity and whose kernels do not run (fake_cudart.cpp)."""
import ctypes
import importlib.util
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_1406_7635_gb300")
MM_ERR_OOM, MM_ERR_STATE = -3, -7


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """The binding over the library with the test's runtime; .rt its controls."""
    from paper_1406_7635_gb300 import build as b
    b.build()
    objs = [os.path.join(b.OUT, u.replace(".cu", ".o")) for u in b.UNITS]
    if not all(os.path.exists(o) for o in objs):
        b.build(force=True)
    lib = str(tmp_path_factory.mktemp("fake") / "libmm_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(b._nvcc())), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I" + cuda, "-o", lib,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    spec = importlib.util.spec_from_file_location("paper_1406_7635_gb300.mm_fake", os.path.join(PKG, "mm.py"))
    mod = importlib.util.module_from_spec(spec)
    keep, b.LIB = b.LIB, lib
    try:
        spec.loader.exec_module(mod)
    finally:
        b.LIB = keep
    rt = mod._lib
    rt.fake_set_capacity.argtypes = [ctypes.c_size_t]
    rt.fake_fail_at.argtypes = [ctypes.c_longlong]
    rt.fake_used.restype = rt.fake_peak.restype = ctypes.c_size_t
    rt.fake_launched.restype = ctypes.c_char_p
    mod.rt = rt
    return mod


@pytest.fixture(autouse=True)
def unlimited(fake):
    def free():
        fake.rt.fake_set_capacity((1 << 64) - 1)
        fake.rt.fake_fail_at(-1)
        fake.rt.fake_no_cooperative(0)
        fake.rt.fake_launched()
    free()
    yield
    free()


def kernels(fake):
    return fake.rt.fake_launched().decode()


def context(fake, shape):
    ctx = fake.Context(*shape, 2e-9, 2e-9, 2e-9)
    ctx.set_material(0, 8e5, 1.3e-11, 0.1)
    m = np.zeros((3,) + ctx.shape, np.float32)
    m[0] = 1.0
    ctx.set_m(m)
    return ctx


def field_calls(fake, ctx):
    n = np.zeros((3,) + ctx.shape, np.float32)
    p = n.ctypes.data_as(ctypes.c_void_p)
    return [lambda: ctx.step(1), lambda: ctx.run(1e-12), ctx.get_bdemag, ctx.get_beff, ctx.get_torque, ctx.get_energies,
            ctx.get_max_torque, lambda: ctx.set_yz_kernels(1), lambda: ctx.profile_attempts(1), lambda: ctx.relax(10),
            lambda: fake._check(fake.mm_demag_apply(ctx.h, p, p))]


# a film and a thin stack (persistent kernel), a cluster grid, a large grid
@pytest.mark.parametrize("shape", [(64, 16, 1), (32, 32, 4), (32, 32, 16), (32, 20, 64)])
@pytest.mark.parametrize("pbc", [(1, 0, 0), (0, 0, 0)])
def test_a_failed_set_pbc_leaves_an_error_not_a_stale_plan(fake, shape, pbc):
    """Whichever of its allocations fails, a context whose set_pbc failed runs
    no kernel until a later set_pbc succeeds: its buffers and its film plan
    are not those of its grid."""
    ctx = context(fake, shape)
    failed = 0
    for k in range(40):
        fake.rt.fake_fail_at(k)
        try:
            ctx.set_pbc(*pbc)
        except fake.MMError as e:
            assert e.code == MM_ERR_OOM
            fake.rt.fake_fail_at(-1)
            kernels(fake)
            for call in field_calls(fake, ctx):
                with pytest.raises(fake.MMError) as ei:
                    call()
                assert ei.value.code == MM_ERR_STATE
            assert kernels(fake) == ""
            ctx.get_m()              # (the state is there)
            failed += 1
        fake.rt.fake_fail_at(-1)
        ctx.set_pbc(*pbc)            # succeeds again
        ctx.step(1)
        ctx.get_bdemag()
    assert failed >= 5               # spectrum, octant and the tensor's work space
    ctx.close()


def make(fake, kind):
    """The allocations of one creation, which is closed again."""
    if kind == "context":
        obj = fake.Context(40, 40, 9, 2e-9, 2e-9, 2e-9)
    elif kind == "film":
        obj = fake.Context(64, 40, 1, 2e-9, 2e-9, 2e-9)
    elif kind == "batch":
        obj = fake.Batch([dict(nx=32, ny=16, nz=nz, dx=2e-9, dy=2e-9, dz=2e-9, msat=8e5, aex=1e-11, alpha=0.1,
                               bext=(0, 0, 0)) for nz in (1, 2)])
    else:
        obj = fake.FNO(32, 32, width=32, layers=2, modes_x=8, modes_y=8, max_batch=2)
    obj.close()


@pytest.mark.parametrize("kind", ["context", "film", "batch", "network"])
def test_a_failed_creation_keeps_nothing(fake, kind):
    """MM_ERR_OOM at creation gives everything back, its error included: the
    next creation in the same thread succeeds."""
    base, failed = fake.rt.fake_used(), 0
    for k in range(80):
        fake.rt.fake_fail_at(k)
        try:
            make(fake, kind)
        except fake.MMError as e:
            assert e.code == MM_ERR_OOM
            failed += 1
        assert fake.rt.fake_used() == base
        fake.rt.fake_fail_at(-1)
        make(fake, kind)
    assert failed > 10


# kernels of a large grid (the three (y, z) kernels, the row-stage kernels)
FAST = ("k_zk", "k_rs_")


@pytest.mark.parametrize("nx,ny,nz", [(20, 18, 64), (17, 21, 33)])
def test_a_large_grid_without_room_for_its_kernels_takes_the_general_ones(fake, nx, ny, nz):
    """At creation and in set_pbc: a failure of any allocation that the
    general convolution does without leaves a working context, all of them
    given back; a failure of any other is MM_ERR_OOM, nothing kept."""
    base = fake.rt.fake_used()
    ctx = context(fake, (nx, ny, nz))
    full = fake.rt.fake_used() - base
    kernels(fake)
    ctx.step(1)
    ctx.get_bdemag()
    names = kernels(fake)
    assert all(f in names for f in FAST)
    ctx.close()
    assert fake.rt.fake_used() == base
    up = lambda n: 1 << (2 * n - 2).bit_length()  # noqa: E731
    hx, hy, hz = up(nx) // 2 + 1, up(ny) // 2 + 1, up(nz) // 2 + 1
    extra = [8 * 3 * hx * nz * up(ny), 24 * hx * hy * hz, 12 * nx * ny * nz, 12 * nx * ny * nz]
    general = 0
    for k in range(60):
        fake.rt.fake_fail_at(k)
        try:
            ctx = context(fake, (nx, ny, nz))
        except fake.MMError as e:
            assert e.code == MM_ERR_OOM and fake.rt.fake_used() == base
            continue
        used = fake.rt.fake_used() - base
        if used != full:
            general += 1
            assert used == full - sum(extra)
            for _ in range(2):
                kernels(fake)
                ctx.step(1)
                ctx.get_bdemag()
                names = kernels(fake)
                assert not any(f in names for f in FAST) and "k_fx" in names
                assert ctx.set_yz_kernels(0) == 0 and ctx.set_yz_kernels(1) == 0
            fake.rt.fake_fail_at(-1)
            ctx.set_pbc(0, 0, 0)     # room again: the fast kernels
            assert fake.rt.fake_used() - base == full
            ctx.step(1)
            names = kernels(fake)
            assert all(f in names for f in FAST)
        ctx.close()
    assert general == len(extra)
    # set_pbc
    ctx = context(fake, (nx, ny, nz))
    general = 0
    for k in range(20):
        fake.rt.fake_fail_at(k)
        try:
            ctx.set_pbc(0, 0, 0)
        except fake.MMError:
            continue
        if fake.rt.fake_used() - base != full:
            general += 1
            assert fake.rt.fake_used() - base == full - sum(extra)
            ctx.step(1)
    assert general == len(extra)
    ctx.close()


@pytest.mark.parametrize("shape", [(64, 16, 1), (32, 32, 4)])
def test_a_refused_cooperative_launch_steps_with_the_stage_kernels(fake, shape):
    """A stream on fewer multiprocessors than the film kernel's blocks need (a
    partition of the device) refuses its launch: the call runs on the stage
    kernels' graph, which needs no co-residency, and so do later ones."""
    ctx = context(fake, shape)
    kernels(fake)
    ctx.step(1)
    assert "k_film" in kernels(fake)
    fake.rt.fake_no_cooperative(1)
    for call in (lambda: ctx.step(1), lambda: ctx.run(1e-12)):
        call()
        names = kernels(fake)
        assert "graph" in names and "k_film" not in names
    ctx.get_bdemag()             # (the refusal is no error of a later call)
    ctx.close()


def test_a_batch_holds_eleven_vectors_per_instance(fake):
    """m twice, seven slopes, and two buffers that are in turn the input and
    the field of a stage, beside the spectrum."""
    def held(n):
        base = fake.rt.fake_used()
        b = fake.Batch([dict(nx=96, ny=96, nz=4, dx=2e-9, dy=2e-9, dz=2e-9, msat=8e5, aex=1e-11, alpha=0.1,
                             bext=(0, 0, 0))] * n)
        used = fake.rt.fake_used() - base
        b.close()
        return used

    vec, spec, small = 12 * 96 * 96 * 4, 8 * 3 * 129 * 4 * 96, 1 << 16
    history = 8 * 4096
    assert 11 * vec + spec <= held(3) - held(2) <= 11 * vec + spec + history + small


def test_a_network_without_room_for_partial_sums_keeps_the_separate_products(fake):
    """The fused backward pass needs a buffer that the separate products do
    without: no room for it is no reason to refuse the network."""
    u = np.zeros((2, 3, 32, 32), np.float32)
    p = u.ctypes.data_as(ctypes.c_void_p)
    created, fused = 0, []
    for k in range(60):
        fake.rt.fake_fail_at(k)
        try:
            net = fake.FNO(32, 32, width=32, layers=2, modes_x=8, modes_y=8, max_batch=2)
        except fake.MMError as e:
            assert e.code == MM_ERR_OOM
            continue
        fake.rt.fake_fail_at(-1)
        kernels(fake)
        g = np.zeros(net.nparams(), np.float32)
        loss = ctypes.c_double()
        for _ in range(2):
            fake._check(fake.mm_fno_grad(net.h, p, p, 2, g.ctypes.data_as(ctypes.c_void_p), ctypes.byref(loss)))
        fused.append("k_bwd_pw" in kernels(fake))
        net.close()
        created += 1
    assert created > 10 and fused.count(False) == 1 and not fused[0]


def test_a_longer_replay_sequence_without_room_keeps_the_one_there(fake):
    base = fake.rt.fake_used()
    ctx = context(fake, (20, 20, 5))
    ctx.set_fixed_dt_sequence([1e-14] * 4)
    held = fake.rt.fake_used()
    fake.rt.fake_fail_at(0)
    with pytest.raises(fake.MMError) as ei:
        ctx.set_fixed_dt_sequence([1e-14] * 1000)
    assert ei.value.code == MM_ERR_OOM
    assert fake.rt.fake_used() == held      # (steps still replay from the buffer that is there)
    ctx.step(1)
    ctx.get_bdemag()                        # (no error left for a later call)
    ctx.set_fixed_dt_sequence([1e-14] * 1000)
    assert fake.rt.fake_used() == held + 8 * 996
    ctx.close()
    assert fake.rt.fake_used() == base


def test_no_room_in_a_call_is_no_error_of_the_next(fake):
    """Calls that allocate on the way: the (y, z) buffer asked for, the table
    of the spin torques, the surrogate's accumulators and its training pairs.
    Each reports MM_ERR_OOM and the context steps on; training puts m back."""
    ctx = context(fake, (32, 32, 16))
    ctx.set_yz_kernels(1)
    net = fake.FNO(16, 40, width=8, layers=1, modes_x=4, modes_y=4, max_batch=2)
    film = context(fake, (40, 16, 1))
    film.set_material(0, 8e5, 1.3e-11, 0.1, jcur=(1e12, 0.0, 0.0), xi=0.05)
    film.step(1)
    m = film.get_m()

    def torque():
        film.enable_stt(True, False)
        film.step(1)

    calls = [(lambda: ctx.set_yz_kernels(2), ctx), (torque, film),
             (lambda: film.set_demag_surrogate(net, 8e5), film),
             (lambda: film.train_surrogate(net, 8e5, 2, 1, 0, 0.0, 1, 1, 1e-3), film)]
    for call, c in calls:
        for k in range(6):
            fake.rt.fake_fail_at(k)
            try:
                call()
            except fake.MMError as e:
                assert e.code == MM_ERR_OOM
            else:
                break
            fake.rt.fake_fail_at(-1)
            assert np.array_equal(film.get_m(), m)
            ctx.step(1)
            ctx.get_bdemag()
            film.set_m(m)
        else:
            raise AssertionError("more allocations than expected")
        fake.rt.fake_fail_at(-1)
        assert k > 0
        film.set_demag_surrogate(None, 8e5)
    for c in (ctx, film, net):
        c.close()
