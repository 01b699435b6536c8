"""The sweeps themselves, one per step, as lbm_set_streaming asks for them: small
lattices take several steps per launch otherwise, and then rows per block, prefetch
distance and the order of row bands matter to a call's last step alone."""
import numpy as np
import pytest

from paper_1909_13086_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

TWO, ONE = lbm.LBM_STREAM_TWO_BUFFERS, lbm.LBM_STREAM_ONE_BUFFER


@pytest.fixture(scope="module")
def stream():
    import torch

    torch.cuda.set_device(0)
    return torch.cuda.Stream().cuda_stream


@pytest.mark.parametrize("mode", [TWO, ONE])
@pytest.mark.parametrize("prec", ["fp32", "bf16sr", "fp64"])
def test_launch_shape_does_not_change_populations(stream, prec, mode):
    nx, ny, p = 260, 45, workloads.params(Ra=1e5)
    ref = None
    for rows, pf in ((1, 0), (1, 4), (3, 2), (8, 64)):
        lat = lbm.Lattice(nx, ny, p, precision=prec, stream=stream)
        lbm.lbm_set_streaming(lat.h, mode)
        lbm.lbm_set_launch(lat.h, rows, pf, 16)
        lat.step(120)
        f, g, _ = lat.populations()
        if ref is None:
            ref = (f, g)
        else:
            assert np.array_equal(f, ref[0]) and np.array_equal(g, ref[1]), (rows, pf)


@pytest.mark.parametrize("mode", [TWO, ONE])
@pytest.mark.parametrize("problem", ["cavity", "stefan"])
@pytest.mark.parametrize("ny", [3, 4, 5, 7, 10])
def test_row_bands_in_both_directions(orc, stream, problem, ny, mode):
    """Every band count (1 to 10, a ragged last band) in both directions (odd and even
    steps) against the oracle: FP64 fields to 1e-12 of their scale."""
    nx = 130
    p = (workloads.params(Ra=1e5, strip_center=0.45, strip_width=0.3) if problem == "cavity"
         else workloads.stefan_1024x4(Ste=1.0, nx=nx)[2])
    ref = orc.Oracle(nx, ny, **p)
    ref.step(9)
    want = ref.fields()
    for rows in (1, 2, 3, 4):
        lat = lbm.Lattice(nx, ny, p, precision="fp64", stream=stream)
        lbm.lbm_set_streaming(lat.h, mode)
        lbm.lbm_set_launch(lat.h, rows, 2, 0)
        lat.step(9)
        got = lat.fields()
        for k in ("H", "T", "fl", "ux", "uy", "rho"):
            scale = max(np.abs(want[k]).max(), 0.1 / 3 ** 0.5 if k in ("ux", "uy") else 1.0)
            assert np.abs(got[k] - want[k]).max() <= 1e-12 * scale, (rows, k)
        assert lat.diagnostics()["Q_cum"] == pytest.approx(ref.diagnostics()["Q_cum"], rel=1e-12, abs=1e-15)
        lat.close()


@pytest.mark.parametrize("mode", [TWO, ONE])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_graph_replay_matches_direct_launches(stream, prec, mode):
    nx, ny, p = 300, 77, workloads.params(Ra=1e5, strip_center=0.4)
    out = []
    for chunk, diag_every in ((0, 0), (128, 0), (0, 50), (32, 50), (7, 3)):
        lat = lbm.Lattice(nx, ny, p, precision=prec, stream=stream)
        lbm.lbm_set_streaming(lat.h, mode)
        lbm.lbm_set_launch(lat.h, 1, 4, chunk)
        lbm.lbm_set_diag_every(lat.h, diag_every)
        lat.step(413)
        lat.step(290)
        out.append((*lat.populations(), lat.diagnostics()))
    for f, g, s, d in out[1:]:
        assert s == out[0][2] == 703 and d == out[0][3]
        assert np.array_equal(f, out[0][0]) and np.array_equal(g, out[0][1])


@pytest.mark.parametrize("mode", [TWO, ONE])
@pytest.mark.parametrize("rows,prefetch,interleave", [(1, 0, 1), (4, 16, 1), (1, 4, 0), (3, 8, 0)])
def test_batch_launch_shapes_equal_solo(stream, rows, prefetch, interleave, mode):
    cases = [(256, 128, dict(Ra=1e6, strip_center=c, seed=k)) for k, c in enumerate((0.2, 0.5, 0.8))]
    solo, members = ([lbm.Lattice(nx, ny, workloads.params(**kw), precision="fp32", stream=stream) for nx, ny, kw in cases]
                     for _ in range(2))
    for lat in solo:
        lbm.lbm_set_streaming(lat.h, TWO)
        lat.step(130)
    b = lbm.Batch(4, stream)
    for lat in members:
        b.add(lat)
    lbm.lbm_batch_set_streaming(b.b, mode)
    lbm.lbm_batch_set_launch(b.b, rows, prefetch, interleave)
    b.step(130)
    b.close()
    for s, m in zip(solo, members):
        for x, y in zip(s.populations(), m.populations()):
            assert np.array_equal(x, y)
        assert s.diagnostics() == m.diagnostics()


@pytest.mark.parametrize("calls,n", [(1, 5), (3, 20)])
def test_full_size_default_path_vs_oracle_fp32(orc, stream, calls, n):
    """2048 x 1024 production cavity, FP32, as the library runs it (two steps per pass
    over memory, diagnostics every 20th step): from the GPU's own populations after 100
    steps, direct and replayed pieces against the oracle's steps, every population of
    every cell, and the fields."""
    nx, ny, p = workloads.cavity_2048x1024()
    lat = lbm.Lattice(nx, ny, p, precision="fp32", stream=stream)
    lbm.lbm_set_diag_every(lat.h, 20)
    lat.step(100)
    f0, g0, s0 = lat.populations()
    ref = orc.Oracle(nx, ny, threads=8, **p)
    ref.set_populations(f0, g0, s0)
    del f0, g0
    before = lbm.lbm_get_kernel_launches(lat.h)
    for _ in range(calls):
        lat.step(n)
    # pairs of plain steps, an odd one alone, and the diagnostic sweep with its fold
    assert lbm.lbm_get_kernel_launches(lat.h) - before == calls * ((n - 1) // 2 + (n - 1) % 2 + 2)
    ref.step(calls * n)
    f1, g1, s1 = lat.populations()
    fo, go = ref.populations()
    assert s1 == s0 + calls * n
    assert np.abs(g1 - go).max() <= 1e-5
    assert np.abs(f1 - fo).max() <= 1e-5
    del f1, g1, fo, go
    F, Fo = lat.fields(), ref.fields()
    for name in ("T", "fl", "ux", "uy"):
        assert np.abs(F[name] - Fo[name]).max() <= 1e-5, name
