"""Several steps per launch (tiles in shared memory, bands of two steps, their
batch forms) against one two-buffer sweep per step, which lbm_set_streaming asks
for: populations, diagnostics, fields and history bitwise, at sizes around the
edges of cores, strips and bands, at step counts that leave remainders, in every
storage type the kernels take, with rates other than 1."""
import numpy as np
import pytest

from paper_1909_13086_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    import torch

    torch.cuda.set_device(0)
    return torch.cuda.Stream().cuda_stream


def start(nx, ny, p, prec, stream, seed=3):
    lat = lbm.Lattice(nx, ny, p, precision=prec, stream=stream)
    f, g = workloads.random_populations(nx, ny, seed)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    lat.set_populations(w * (1 + 5.0 * (f - 1 / 9)), g, 0)
    lbm.lbm_set_history(lat.h, 256)
    return lat


def state(lat):
    f, g, step = lat.populations()
    h = lbm.lbm_read_history(lat.h, 256)
    return [f, g, step, *[v for _, v in sorted(lat.diagnostics(raise_on_diverged=False).items())],
            *[v for _, v in sorted(lat.fields().items())], *[h[k] for k in sorted(h)]]


def assert_same(a, b, what):
    for k, (x, y) in enumerate(zip(state(a), state(b))):
        assert np.array_equal(np.asarray(x), np.asarray(y), equal_nan=True), (what, k)


def compare(nx, ny, p, prec, stream, calls, diag_every=0):
    lat, ref = (start(nx, ny, p, prec, stream) for _ in range(2))
    lbm.lbm_set_streaming(ref.h, lbm.LBM_STREAM_TWO_BUFFERS)
    for n in calls:
        for L in (lat, ref):
            lbm.lbm_set_diag_every(L.h, diag_every)
            L.step(n)
        assert_same(lat, ref, (nx, ny, prec, n))


RATES = dict(k0=0.9, k0f=1.1, k1f=1.2)


@pytest.mark.parametrize("prec", ["fp32", "bf16sr", "fp16"])
@pytest.mark.parametrize("nx,ny", [(2, 2), (2, 40), (31, 3), (33, 17), (64, 32), (65, 33), (257, 129), (700, 90)])
def test_tiles(stream, prec, nx, ny):
    compare(nx, ny, workloads.params(Ra=1e5, strip_center=0.4, **RATES), prec, stream, (2, 3, 18, 33, 33, 33), 9)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16sr", "bf16"])
@pytest.mark.parametrize("problem,nx,ny", [("stefan", 2, 2), ("stefan", 17, 4), ("stefan", 300, 32), ("stefan", 40, 33),
                                           ("cavity", 33, 17), ("cavity", 130, 70)])
def test_tiles_without_flow(stream, prec, problem, nx, ny):
    if problem == "stefan":
        p = workloads.stefan_1024x4(Ste=0.5, nx=nx)[2]
    else:
        p = workloads.params(Ra=1e5, flow_on=0, strip_width=0.6)
    compare(nx, ny, p, prec, stream, (2, 3, 18, 33))


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16sr"])
@pytest.mark.parametrize("nx,ny", [(3, 2), (40, 5), (130, 32)])
def test_tiles_of_a_periodic_lattice_with_flow(stream, prec, nx, ny):
    p = workloads.params(problem=workloads.STEFAN, Ra=1e4, alpha_override=0.05, **RATES)
    compare(nx, ny, p, prec, stream, (2, 3, 18, 33))


@pytest.mark.parametrize("nx,ny", [(1023, 520), (1025, 513), (8, 65535), (4500, 130), (2048, 1024)])
def test_bands(stream, nx, ny):
    compare(nx, ny, workloads.params(Ra=1e6, strip_center=0.6, **RATES), "fp32", stream, (2, 3, 10, 10, 11), 4)


MEMBERS = [(256, 128, dict(Ra=1e6, strip_center=0.2)), (300, 77, dict(Ra=1e5, strip_center=0.65)), (64, 32, dict()),
           (3, 5, dict(Ra=1e4)), (131, 9, dict(Ra=1e6, strip_width=0.4))]


@pytest.mark.parametrize("prec", ["fp32", "bf16sr"])
@pytest.mark.parametrize("copies", [1, 14])
def test_batches(stream, prec, copies):
    """Few small members (tiles) and many (bands), one of them a step ahead;
    odd and even calls, pieces direct and replayed."""
    groups = []
    for mode in (None, lbm.LBM_STREAM_TWO_BUFFERS):
        lats = [start(nx, ny, workloads.params(**RATES, **kw), prec, stream, seed=k)
                for k, (nx, ny, kw) in enumerate(MEMBERS * copies)]
        lats[1].step(1)
        b = lbm.Batch(len(lats), stream)
        for lat in lats:
            b.add(lat)
        if mode is not None:
            lbm.lbm_batch_set_streaming(b.b, mode)
        for n in (1, 2, 3, 20, 135, 20, 135, 20):
            b.step(n)
        b.close()
        groups.append(lats)
    for k, (x, y) in enumerate(zip(*groups)):
        assert_same(x, y, (prec, copies, k))


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_static_step_takes_buffers_on_any_element(offset):
    """lbm_step_static's FP32 buffers need no alignment beyond an element's: the
    sweep with 8-byte accesses serves the aligned ones, one value at a time the
    others; same populations and diagnostics."""
    import torch

    nx, ny = 130, 40
    p = workloads.params(Ra=1e5, strip_center=0.4)
    n = 2 * ny * 18 * 128
    gen = torch.Generator().manual_seed(1)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).repeat(2)[None, None, :, None]
    src = (w * (1 + 0.05 * torch.rand(2, ny, 18, 128, generator=gen))).float().reshape(-1).cuda()
    out = []
    s = torch.cuda.Stream()
    for k in (0, offset):
        bufs = [torch.zeros(n + 4, device="cuda") for _ in range(2)]
        bufs[0][k:k + n] = src
        torch.cuda.synchronize()
        d = lbm.lbm_step_static(bufs[0].data_ptr() + 4 * k, bufs[1].data_ptr() + 4 * k, nx, ny, lbm.LBM_FP32, p, 0,
                                s.cuda_stream)
        out.append((bufs[1][k:k + n].cpu().numpy(), d))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("nx,ny", [(512, 256), (256, 128)])
def test_fields_into_separate_pinned_arrays(stream, nx, ny):
    """Six pinned arrays of a power-of-two size usually follow one another in
    memory without being one allocation; a copy may not span two of them."""
    import torch

    lat = lbm.Lattice(nx, ny, workloads.params(Ra=1e6), precision="fp32", stream=stream)
    lat.step(5)
    want = lat.fields()
    pinned = [torch.empty(ny, nx, dtype=torch.float64, pin_memory=True).numpy() for _ in range(6)]
    lbm.lbm_read_fields(lat.h, 63, *sorted(pinned, key=lambda a: a.ctypes.data))
    for name, got in zip(lbm.FIELD_NAMES, sorted(pinned, key=lambda a: a.ctypes.data)):
        assert np.array_equal(got, want[name]), name


@pytest.mark.parametrize("prec,problem,kw,nx,ny", [
    ("fp64", "cavity", {}, 64, 32), ("fp64", "cavity", dict(flow_on=0), 33, 17), ("fp64", "stefan", {}, 300, 4),
    ("fp32", "cavity", {}, 65, 33), ("fp32", "cavity", dict(flow_on=0), 130, 70), ("fp32", "stefan", {}, 300, 32),
    ("bf16sr", "cavity", {}, 31, 3), ("bf16sr", "stefan", {}, 17, 4), ("fp16", "cavity", dict(flow_on=0), 64, 32)])
def test_batch_of_one(stream, prec, problem, kw, nx, ny):
    """One member, of every kind, whether or not the batch kernels take several
    steps of it: the member alone, one sweep per step, over odd and even calls."""
    p = workloads.stefan_1024x4(Ste=0.5, nx=nx)[2] if problem == "stefan" else workloads.params(Ra=1e5, **RATES, **kw)
    lat, ref = (start(nx, ny, p, prec, stream) for _ in range(2))
    lbm.lbm_set_streaming(ref.h, lbm.LBM_STREAM_TWO_BUFFERS)
    b = lbm.Batch(1, stream)
    b.add(lat)
    for n in (1, 3, 20, 135, 3, 135):
        b.step(n)
        ref.step(n)
        for x, y in zip(lat.populations(), ref.populations()):
            assert np.array_equal(x, y), (prec, problem, n)
        for k, v in ref.fields().items():
            assert np.array_equal(lat.fields()[k], v), (prec, problem, n, k)
    b.close()


@pytest.mark.parametrize("every", [1, 2, 3, 4, 5])
def test_bands_between_frequent_diagnostics(stream, every):
    """Pieces too short for bands, or with an odd plain step: swept in place except for
    the call's last; the fields of the step before are there after every call."""
    compare(1025, 513, workloads.params(Ra=1e6, strip_center=0.6, **RATES), "fp32", stream, (1, 2, 3, 4, 12, 12, 13, 12),
            every)


@pytest.mark.parametrize("prec", ["fp32", "bf16sr"])
def test_batch_bands_in_several_waves(stream, prec):
    """1200 members of 40 x 30: more bands than blocks that run at once."""
    groups = []
    for mode in (None, lbm.LBM_STREAM_TWO_BUFFERS):
        lats = [lbm.Lattice(40, 30, workloads.params(Ra=1e5, strip_center=0.2 + 0.0005 * k, seed=k, init_amp=0.1, **RATES),
                            precision=prec, stream=stream) for k in range(1200)]
        b = lbm.Batch(len(lats), stream)
        for lat in lats:
            b.add(lat)
        if mode is not None:
            lbm.lbm_batch_set_streaming(b.b, mode)
        for n in (3, 20, 7):
            b.step(n)
        b.close()
        groups.append([lat.populations() for lat in lats[::173]])
    for x, y in zip(*groups):
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1]) and x[2] == y[2] == 30


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16", "fp16sr", "bf16sr"])
@pytest.mark.parametrize("nx", [2, 3, 33, 64, 65, 129, 160, 161])
def test_narrow_lattices_by_every_path(stream, prec, nx):
    """Widths around those where sweeps take one cell per thread: several steps per
    launch, one buffer and two buffers end in the same bits."""
    p = workloads.params(Ra=1e5, strip_center=0.4, strip_width=0.5, **RATES)
    lats = [start(nx, 37, p, prec, stream) for _ in range(3)]
    lbm.lbm_set_streaming(lats[1].h, lbm.LBM_STREAM_ONE_BUFFER)
    lbm.lbm_set_streaming(lats[2].h, lbm.LBM_STREAM_TWO_BUFFERS)
    for n in (1, 2, 7, 20, 7, 20):
        for lat in lats:
            lbm.lbm_set_diag_every(lat.h, 5)
            lat.step(n)
        assert_same(lats[0], lats[2], (prec, nx, n))
        assert_same(lats[1], lats[2], (prec, nx, n))


def test_modes_in_turn(stream):
    """lbm_set_streaming between calls, LBM_STREAM_AUTO among the modes: a lattice and a
    batch go on from the same state whatever moved it there."""
    p = workloads.params(Ra=1e6, strip_center=0.4)
    for prec in ("fp32", "fp16sr", "fp64"):
        lat, ref = (start(130, 70, p, prec, stream) for _ in range(2))
        members = [start(64, 32, p, prec, stream, seed=k) for k in range(2)]
        refs = [start(64, 32, p, prec, stream, seed=k) for k in range(2)]
        lbm.lbm_set_streaming(ref.h, lbm.LBM_STREAM_TWO_BUFFERS)
        batch, batch_ref = lbm.Batch(2, stream), lbm.Batch(2, stream)
        for b, ms in ((batch, members), (batch_ref, refs)):
            for m in ms:
                b.add(m)
        lbm.lbm_batch_set_streaming(batch_ref.b, lbm.LBM_STREAM_TWO_BUFFERS)
        for mode in (lbm.LBM_STREAM_ONE_BUFFER, lbm.LBM_STREAM_AUTO, lbm.LBM_STREAM_TWO_BUFFERS, lbm.LBM_STREAM_AUTO):
            lbm.lbm_set_streaming(lat.h, mode)
            lbm.lbm_batch_set_streaming(batch.b, mode)
            for n in (7, 20, 20):
                for x in (lat, ref, batch, batch_ref):
                    x.step(n)
        assert_same(lat, ref, prec)
        for x, y in zip(members, refs):
            assert_same(x, y, prec)
        batch.close()
        batch_ref.close()
    for bad in (-2, 2):
        with pytest.raises(lbm.LbmError):
            lbm.lbm_set_streaming(lat.h, bad)


def test_autotuners_time_what_runs(stream):
    """Where several steps share a launch the tuners leave the sweeps' shape alone and
    return the time of the kernels that run: far less than a sweep per step takes here."""
    p = workloads.params(Ra=1e6, strip_center=0.35)
    lat, swept = (lbm.Lattice(260, 126, p, precision="fp32", stream=stream) for _ in range(2))
    lbm.lbm_set_launch(lat.h, 7, 5, 64)
    lbm.lbm_set_streaming(swept.h, lbm.LBM_STREAM_ONE_BUFFER)
    t, ts = lbm.lbm_autotune(lat.h, 100), lbm.lbm_autotune(swept.h, 100)
    assert (t["rows"], t["prefetch"]) == (7, 5) and ts["rows"] in (1, 2, 3, 4)
    assert 0 < 1.5 * t["us_per_step"] < ts["us_per_step"]
    lbm.lbm_set_streaming(swept.h, lbm.LBM_STREAM_AUTO)
    assert lbm.lbm_autotune(swept.h, 100)["us_per_step"] == 0.0  # the same kind as the first now
    us = []
    for mode in (lbm.LBM_STREAM_AUTO, lbm.LBM_STREAM_TWO_BUFFERS):
        b = lbm.Batch(2, stream)
        members = [lbm.Lattice(260, 126, p, precision="fp32", stream=stream) for _ in range(2)]
        for m in members:
            b.add(m)
        lbm.lbm_batch_set_streaming(b.b, mode)
        if mode == lbm.LBM_STREAM_AUTO:
            lbm.lbm_batch_set_launch(b.b, 3, 2, 1)
        t = lbm.lbm_batch_autotune(b.b, 100)
        if mode == lbm.LBM_STREAM_AUTO:
            assert (t["rows"], t["prefetch"], t["interleave"]) == (3, 2, 1)
        us.append(t["us_per_step"])
        b.close()
    assert 0 < 1.5 * us[0] < us[1]


@pytest.mark.parametrize("diag_every,per_call", [(0, 4 + 1 + 2), (4, 4 * 2 + 1 + 2), (1, 10 * 2)])
def test_kernel_launches_are_counted(stream, diag_every, per_call):
    """A call of 10 steps, launched directly, captured and replayed.  Bands: four
    pairs, an odd step, a diagnostic sweep and its fold; diagnostics every 4th step: two
    pieces of a pair, an odd step, a sweep and a fold, then one step and a sweep and a
    fold; every step: ten sweeps and folds.  Two buffers: a sweep per step, a fold."""
    p = workloads.params(Ra=1e6, strip_center=0.6)
    lat, ref = (lbm.Lattice(1025, 513, p, precision="fp32", stream=stream) for _ in range(2))
    lbm.lbm_set_diag_every(lat.h, diag_every)
    lbm.lbm_set_streaming(ref.h, lbm.LBM_STREAM_TWO_BUFFERS)
    for call in range(1, 4):
        # each call starts at a multiple of diag_every
        lat.set_populations(*lat.populations()[:2], 0)
        before = lbm.lbm_get_kernel_launches(lat.h)
        lat.step(10)
        assert lbm.lbm_get_kernel_launches(lat.h) - before == per_call
        ref.step(10)
        assert lbm.lbm_get_kernel_launches(ref.h) == 11 * call


def test_kernel_launches_of_a_batch_are_counted(stream):
    p = workloads.params(Ra=1e5)
    for prec, members, want in (("fp32", 60, 4 + 1 + 2), ("fp64", 2, 11)):
        lats = [lbm.Lattice(128, 128, p, precision=prec, stream=stream) for _ in range(members)]
        b = lbm.Batch(members, stream)
        for lat in lats:
            b.add(lat)
        for call in range(1, 4):
            b.step(10)
            assert lbm.lbm_batch_get_kernel_launches(b.b) == want * call
        b.close()


@pytest.mark.parametrize("rates", [{}, RATES])
@pytest.mark.parametrize("nx,ny", [(2, 2), (31, 3), (33, 17), (64, 32), (65, 33), (181, 181), (256, 128)])
def test_fp64_tiles(stream, rates, nx, ny):
    """With k0 = k0f = 1 the collision drops the terms in the old populations: both
    forms, in tiles and in sweeps."""
    compare(nx, ny, workloads.params(Ra=1e5, strip_center=0.4, **rates), "fp64", stream, (2, 3, 18, 33, 33), 9)


@pytest.mark.parametrize("prec,nx,ny", [("fp32", 64, 32), ("fp64", 64, 32), ("bf16", 65, 33), ("fp32", 1025, 513)])
def test_history_shorter_than_a_launch(stream, prec, nx, ny):
    """A ring of one or three entries wraps inside a launch of several steps."""
    for cap in (1, 3):
        lat, ref = (start(nx, ny, workloads.params(Ra=1e5, strip_center=0.4), prec, stream) for _ in range(2))
        lbm.lbm_set_streaming(ref.h, lbm.LBM_STREAM_TWO_BUFFERS)
        for L in (lat, ref):
            lbm.lbm_set_history(L.h, cap)
        for n in (2, 19, 19, 20):
            for L in (lat, ref):
                L.step(n)
            assert_same(lat, ref, (prec, cap, n))
            assert len(lbm.lbm_read_history(lat.h, 256)["step"]) == min(cap, lat.populations()[2])


@pytest.mark.parametrize("prec,nx,ny", [("fp32", 64, 32), ("fp64", 64, 32), ("bf16sr", 65, 33), ("fp32", 1025, 513)])
def test_no_heated_strip(stream, prec, nx, ny):
    compare(nx, ny, workloads.params(Ra=1e5, strip_width=0.0, **RATES), prec, stream, (2, 3, 18, 18), 9)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("prec,nx,ny", [("fp32", 64, 32), ("fp64", 64, 32), ("fp16", 65, 33), ("bf16sr", 64, 32),
                                        ("fp32", 1025, 513)])
def test_non_finite_populations(stream, prec, nx, ny, bad):
    """A non-finite value spreads through tiles and bands as through sweeps."""
    lat, ref = (start(nx, ny, workloads.params(Ra=1e5), prec, stream) for _ in range(2))
    lbm.lbm_set_streaming(ref.h, lbm.LBM_STREAM_TWO_BUFFERS)
    f, g, _ = lat.populations()
    f[3, ny // 2, nx // 2] = bad
    g[5, 1, 2] = bad
    for L in (lat, ref):
        L.set_populations(f, g, 0)
        L.step(7)
    for x, y in zip(lat.populations(), ref.populations()):
        assert np.array_equal(x, y, equal_nan=True)
    assert lat.diagnostics(raise_on_diverged=False)["nan_flag"] == ref.diagnostics(raise_on_diverged=False)["nan_flag"] == 1


@pytest.mark.parametrize("prec", ["fp16", "fp16sr", "bf16"])
@pytest.mark.parametrize("copies", [1, 14])
def test_batches_of_other_16_bit_types(stream, prec, copies):
    test_batches(stream, prec, copies)


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16", "fp16sr", "bf16sr"])
@pytest.mark.parametrize("nx,ny", [(33, 6101), (129, 3101)])
def test_tall_narrow_lattices_by_every_path(stream, prec, nx, ny):
    """Enough rows for the plain sweeps to take one cell per thread."""
    p = workloads.params(Ra=1e5, strip_center=0.4, strip_width=0.5, **RATES)
    lats = [start(nx, ny, p, prec, stream) for _ in range(3)]
    lbm.lbm_set_streaming(lats[1].h, lbm.LBM_STREAM_ONE_BUFFER)
    lbm.lbm_set_streaming(lats[2].h, lbm.LBM_STREAM_TWO_BUFFERS)
    for lat in lats:
        lbm.lbm_set_diag_every(lat.h, 5)
        for n in (2, 7, 12):
            lat.step(n)
    assert_same(lats[0], lats[2], (prec, nx))
    assert_same(lats[1], lats[2], (prec, nx))
