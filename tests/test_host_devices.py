"""The library's host code on a fake CUDA runtime with two devices (tests/fake/cudart.cpp),
without a GPU: the compiled objects of the build linked with the fake in place of the CUDA
runtime, kernels checked against their launch limits and not run."""
import ctypes as C
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2307_01571_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
KD_DEVICE, KD_HOST = 1, 0


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    objs = [os.path.join(_build.BUILD, o) for _, o, _ in _build.UNITS]
    _build.build(force=not all(os.path.exists(o) for o in objs))
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_build._nvcc())))
    inc = [d for d in glob.glob(os.path.join(cuda, "include")) + glob.glob(os.path.join(cuda, "targets", "*", "include"))
           if os.path.exists(os.path.join(d, "cuda_runtime_api.h"))]
    out = str(tmp_path_factory.mktemp("fake") / "libkd_fake.so")
    r = subprocess.run([shutil.which("g++"), "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-Wl,-z,defs",
                        *[f"-I{d}" for d in inc], os.path.join(HERE, "fake", "cudart.cpp"), *objs, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return C.CDLL(out)


@pytest.fixture
def fake(lib):
    yield lib
    lib.fake_fail_malloc(-1)
    lib.fake_capture_query_error(0)
    lib.fake_refuse_attribute(0)
    lib.fake_set_device(0)


def _net(lib, widths):
    h = C.c_void_p()
    arr = (C.c_int32 * len(widths))(*widths)
    return lib.kd_mlp_create(arr, len(widths) - 1, C.byref(h)), h


def _train(lib, h, batch=8):
    x = np.zeros(1 << 16, np.float32)
    p = C.c_void_p(x.ctypes.data)
    return lib.kd_mlp_train_step(h, p, p, batch, C.c_float(1e-3), None, None)


@pytest.mark.parametrize("precision", [0, 1])
def test_networks_train_on_every_device(fake, precision):
    """The shared-memory limit that the products' kernels need is set on each device that holds
    a network, whichever device held the first one."""
    for dev in (0, 1, 0):
        assert fake.fake_set_device(dev) == 0
        rc, h = _net(fake, [5, 64, 4])
        assert rc == 0
        assert fake.kd_mlp_set_precision(h, precision) == 0
        before = fake.fake_launches()
        assert _train(fake, h) == 0, dev
        assert fake.fake_launches() > before
        fake.kd_mlp_destroy(h)


def test_a_refused_limit_is_not_remembered(fake):
    """A network whose device refuses the limit is not made (or not switched to BF16); later
    ones are."""
    fake.fake_refuse_attribute(1)
    rc, h = _net(fake, [5, 64, 4])
    assert rc != 0 and not h
    fake.fake_refuse_attribute(0)
    rc, h = _net(fake, [5, 64, 4])
    assert rc == 0
    fake.fake_refuse_attribute(1)
    assert fake.kd_mlp_set_precision(h, 1) != 0
    assert _train(fake, h) == 0            # still an FP32 network
    fake.fake_refuse_attribute(0)
    assert fake.kd_mlp_set_precision(h, 1) == 0 and _train(fake, h) == 0
    fake.kd_mlp_destroy(h)


def _sim(lib, nx, ny, precision):
    from paper_2307_01571_gb300 import kd, workloads as W
    wl = W.small(nx, ny, W.GAUSS, units=W.ATOMIC)
    h = C.c_void_p()
    rc = lib.kd_create(C.byref(kd._fill(kd.kd_units, wl.units)), C.byref(kd._fill(kd.kd_grid, wl.grid)),
                       C.byref(kd._fill(kd.kd_field, wl.field)), precision, None, C.byref(h))
    return rc, h, wl


def test_an_error_is_reported_once(fake):
    """A call that failed inside the runtime, or a query whose failure a call gets over, leaves
    nothing behind that a later call's launch check would report as its own."""
    rc, h = _net(fake, [5, 64, 4])
    assert rc == 0
    fake.fake_fail_malloc(0)
    assert _train(fake, h) != 0
    assert fake.fake_last_error() == 0
    made = [_sim(fake, 512, 512, 1) for _ in range(2)]          # together they fill the SMs
    assert all(rc == 0 for rc, _, _ in made)
    fake.fake_capture_query_error(1)
    b = C.c_void_p()
    assert fake.kd_batch_create((C.c_void_p * 2)(*[s for _, s, _ in made]), 2, None, C.byref(b)) == 0
    assert fake.fake_last_error() == 0
    fake.fake_capture_query_error(0)
    assert fake.kd_get_density_x(made[0][1], np.zeros(512).ctypes.data_as(C.c_void_p), KD_HOST) == 0
    fake.kd_batch_destroy(b)
    for _, s, _ in made:
        fake.kd_destroy(s)
    fake.kd_mlp_destroy(h)


# FP64, FP32, FP32 on the tensor cores, double-word; sizes whose sweeps need the raised limit
@pytest.mark.parametrize("precision,nx,ny", [(0, 2048, 1024), (1, 1024, 512), (2, 1024, 64), (3, 1024, 1024)])
def test_simulations_step_on_every_device(fake, precision, nx, ny):
    """As for the networks: the sweeps' limits on both devices."""
    for dev in (0, 1, 0):
        assert fake.fake_set_device(dev) == 0
        rc, h, wl = _sim(fake, nx, ny, precision)
        assert rc == 0, dev
        assert fake.kd_step(h, C.c_double(wl.dt), C.c_int64(3), C.c_int64(0), None, C.c_int64(0), None) == 0, dev
        fake.kd_destroy(h)


def test_persistent_batches_step_on_every_device(fake):
    for dev in (0, 1):
        assert fake.fake_set_device(dev) == 0
        made = [_sim(fake, 512, 64, 1) for _ in range(2)]
        assert all(rc == 0 for rc, _, _ in made)
        b = C.c_void_p()
        assert fake.kd_batch_create((C.c_void_p * 2)(*[h for _, h, _ in made]), 2, None, C.byref(b)) == 0
        assert fake.kd_batch_set_mode(b, 1) == 0
        dt = (C.c_double * 2)(made[0][2].dt, made[0][2].dt)
        assert fake.kd_batch_step(b, dt, C.c_int64(3), C.c_int64(0), None, C.c_int64(0), None) == 0, dev
        fake.kd_batch_destroy(b)
        for _, h, _ in made:
            fake.kd_destroy(h)


def test_batch_buffers_after_a_failed_allocation(fake):
    """Every allocation that a larger batch needs fails in turn: the call reports it, and the
    next calls, at the old batch size and at the new one, use and free no buffer of the old
    set (the fake runtime counts frees of memory that is not live)."""
    for k in range(16):
        rc, h = _net(fake, [5, 64, 64, 4])
        assert rc == 0 and _train(fake, h, 8) == 0
        live = fake.fake_live()
        fake.fake_fail_malloc(k)
        rc = _train(fake, h, 300)
        fake.fake_fail_malloc(-1)
        if rc == 0:             # more than the call allocates
            fake.kd_mlp_destroy(h)
            break
        assert rc == -8, (k, rc)      # KD_ERR_NOMEM
        assert _train(fake, h, 8) == 0 and fake.fake_live() >= live
        assert _train(fake, h, 300) == 0
        fake.kd_mlp_destroy(h)
        assert fake.fake_bad_frees() == 0, k
    assert k > 6 and fake.fake_bad_frees() == 0


def _batch_step(lib, sims, dt):
    b = C.c_void_p()
    assert lib.kd_batch_create((C.c_void_p * len(sims))(*sims), len(sims), None, C.byref(b)) == 0
    rc = lib.kd_batch_step(b, (C.c_double * len(sims))(*[dt] * len(sims)), C.c_int64(2), C.c_int64(0), None, C.c_int64(0), None)
    lib.kd_batch_destroy(b)
    return rc


def test_every_grid_and_variant_has_its_kernels(fake):
    """The kernels that the launch rule names for a grid are among those compiled, for every
    pair of axis lengths and every variant, alone and in a batch that fills the SMs (one that
    is not compiled is refused with an error)."""
    rc, big, _ = _sim(fake, 1024, 512, 1)
    assert rc == 0
    sizes = [1 << k for k in range(2, 13)]
    for nx in sizes:
        for ny in sizes:
            if nx * ny > 1 << 20:
                continue
            rc, h, wl = _sim(fake, nx, ny, 1)
            assert rc == 0, (nx, ny)
            for v in range(4):
                assert fake.kd_set_sweep_variants(h, v, v) == 0, (nx, ny, v)
                assert fake.kd_step(h, C.c_double(wl.dt), C.c_int64(2), C.c_int64(0), None, C.c_int64(0), None) == 0
                assert _batch_step(fake, [h, big], wl.dt) == 0, (nx, ny, v)
            if 16 <= nx <= 512 and 16 <= ny <= 512:
                b = C.c_void_p()
                assert fake.kd_batch_create((C.c_void_p * 1)(h), 1, None, C.byref(b)) == 0
                assert fake.kd_batch_set_mode(b, 1) == 0
                assert fake.kd_batch_step(b, (C.c_double * 1)(wl.dt), C.c_int64(2), C.c_int64(0), None, C.c_int64(0), None) == 0
                fake.kd_batch_destroy(b)
            fake.kd_destroy(h)
    fake.kd_destroy(big)


def test_no_sweep_kernel_is_first_launched_in_a_capture(fake):
    """What a crowded batch launches has run before its graph is captured, whatever variants the
    first member of a shape has and whether a member's variants change after the batch is made."""
    from paper_2307_01571_gb300 import kd, workloads as W
    assert fake.fake_set_device(1) == 0
    rc, big, wl = _sim(fake, 1024, 512, 1)
    assert rc == 0
    sims = [_sim(fake, 128, 64, 1)[1] for _ in range(3)]
    assert fake.kd_set_sweep_variants(sims[0], 2, 3) == 0
    b = C.c_void_p()
    assert fake.kd_batch_create((C.c_void_p * 4)(*sims, big), 4, None, C.byref(b)) == 0
    dt = (C.c_double * 4)(*[wl.dt] * 4)
    # the small kernels of the step loop have no first launch of their own: a lone run's
    assert fake.kd_step(sims[1], C.c_double(wl.dt), C.c_int64(2), C.c_int64(0), None, C.c_int64(0), None) == 0
    before = fake.fake_first_in_capture()
    assert fake.kd_batch_step(b, dt, C.c_int64(2), C.c_int64(0), None, C.c_int64(0), None) == 0
    assert fake.kd_set_sweep_variants(sims[0], 0, 0) == 0
    assert fake.kd_batch_step(b, dt, C.c_int64(2), C.c_int64(0), None, C.c_int64(0), None) == 0
    assert fake.fake_first_in_capture() == before
    fake.kd_batch_destroy(b)
    for s in (*sims, big):
        fake.kd_destroy(s)


@pytest.mark.parametrize("precision", [0, 1])
def test_training_allocates_nothing_at_a_batch_size_already_seen(fake, precision):
    """A step at no more rows than an earlier call's makes no allocation (a stream capture, or a
    device without memory left, allows none), whatever the precision was then."""
    rc, h = _net(fake, [5, 256, 256, 4])
    assert rc == 0
    x = np.zeros(1 << 16, np.float32)
    p = C.c_void_p(x.ctypes.data)
    assert fake.kd_mlp_forward(h, p, 1024, p, KD_DEVICE, None) == 0
    assert fake.kd_mlp_set_precision(h, precision) == 0
    fake.fake_fail_malloc(0)
    for batch in (1024, 700, 300, 8):
        assert _train(fake, h, batch) == 0, batch
    fake.fake_fail_malloc(-1)
    # a change of precision that finds no memory leaves a network that still trains
    fake.fake_fail_malloc(0)
    fake.kd_mlp_set_precision(h, 1 - precision)
    fake.fake_fail_malloc(-1)
    for batch in (8, 1024):
        assert _train(fake, h, batch) == 0
    fake.kd_mlp_destroy(h)
    assert fake.fake_bad_frees() == 0


def test_runs_of_one_shape_capture_their_steps_once(fake):
    """Another time, packet or state is no reason to capture the step loop again; other windows,
    another basis, interval or time step are.  kd_step and kd_batch_step."""
    from paper_2307_01571_gb300 import kd, workloads as W
    rc, h, wl = _sim(fake, 64, 128, 1)
    assert rc == 0
    b = C.c_void_p()
    assert fake.kd_batch_create((C.c_void_p * 1)(h), 1, None, C.byref(b)) == 0
    p = wl.packet
    buf = (kd.kd_obs * 8)()

    def run(packet, t, batch, dt=wl.dt, every=4):
        assert fake.kd_init_packet(h, C.byref(kd._fill(kd.kd_packet, packet))) == 0
        assert fake.kd_set_time(h, C.c_double(t)) == 0
        before = fake.fake_instantiated()
        args = (C.c_int64(12), C.c_int64(every), buf, C.c_int64(12 // every), None)
        rc = fake.kd_batch_step(b, (C.c_double * 1)(dt), *args) if batch else fake.kd_step(h, C.c_double(dt), *args)
        assert rc == 0
        return fake.fake_instantiated() - before

    moved = W.Packet(p.p0x, p.p0y, 0.1 * wl.grid.x_max, 0.0, p.sigma_p, -p.spin, p.basis)
    other_basis = W.Packet(p.p0x, p.p0y, p.r0x, p.r0y, p.sigma_p, p.spin, 1 - p.basis)
    other_window = W.Packet(0.5 * p.p0x, p.p0y, p.r0x, p.r0y, p.sigma_p, p.spin, p.basis)
    for batch in (False, True):
        assert run(p, 0.0, batch) > 0
        for start, t in ((p, 3.0 * wl.dt), (moved, 0.0), (moved, wl.dt), (p, 0.0)):
            assert run(start, t, batch) == 0
        for start, kw in ((other_basis, {}), (other_window, {}), (p, {}), (p, dict(dt=0.5 * wl.dt)), (p, dict(every=6))):
            assert run(start, 0.0, batch, **kw) > 0
            assert run(start, wl.dt, batch, **kw) == 0
    fake.kd_batch_destroy(b)
    fake.kd_destroy(h)
