"""The plans of the kernels that take several steps per launch, made on the host:
which lattices and batches get one."""
import os
import subprocess

import pytest

from paper_1909_13086_gb300 import build, lbm, workloads

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    objs = [os.path.join(build.OBJ, f.replace(".cu", ".o")) for f in build.SOURCES if f != "lbm_api.cu"]
    build.build(force=not all(os.path.exists(o) for o in objs))
    exe = str(tmp_path_factory.mktemp("plans") / "plans")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    os.path.join(HERE, "plans_host.cu"), *objs, "-cudart", "static", "-o", exe], check=True)

    def ask(prec, problem, flow, sizes, streaming=-1):
        line = [lbm.PRECISIONS[prec], problem, flow, streaming, len(sizes), *(v for size in sizes for v in size)]
        out = subprocess.run([exe], input=" ".join(map(str, line)), capture_output=True, text=True, check=True).stdout
        keys = ("w", "h", "t", "threads", "rows")
        v = [int(x) for x in out.split()]
        more = ("tiles", "smem", "prefetch16", "batch_prefetch", "batch_rows", "one", "batch_one", "auto", "batch_auto")
        return dict(zip(keys, v[:5])), dict(zip(keys + more, v[5:]))

    return ask


@pytest.mark.parametrize("n", [1, 2])
@pytest.mark.parametrize("prec,problem,flow,size", [
    ("fp64", workloads.CAVITY, 1, (64, 32)), ("fp64", workloads.CAVITY, 0, (64, 32)),
    ("fp64", workloads.STEFAN, 0, (1024, 4)), ("fp32", workloads.STEFAN, 0, (1024, 4)),
    ("fp32", workloads.STEFAN, 1, (64, 8)), ("fp32", workloads.CAVITY, 0, (256, 128)),
    ("bf16sr", workloads.STEFAN, 0, (300, 32)), ("fp16", workloads.CAVITY, 0, (64, 32))])
def test_a_batch_without_a_several_step_kernel_gets_no_plan(plans, n, prec, problem, flow, size):
    """The batch kernels take cavities with flow in FP32 arithmetic; each of these
    lattices has a plan when stepped alone, and none in a batch, of one member too."""
    batch, solo = plans(prec, problem, flow, [size] * n)
    assert solo["t"] >= 2
    assert batch["t"] == 0 and batch["threads"] == 0


@pytest.mark.parametrize("prec", ["fp32", "bf16sr"])
def test_a_batch_of_one_cavity_gets_the_lattices_plan(plans, prec):
    batch, solo = plans(prec, workloads.CAVITY, 1, [(64, 32)])
    assert batch.items() <= solo.items() and batch["t"] >= 2


@pytest.mark.parametrize("problem,flow,sizes", [
    (workloads.CAVITY, 1, [(2, 2), (64, 32), (100, 50), (128, 64), (181, 181), (256, 128), (1024, 32), (4096, 8)]),
    (workloads.CAVITY, 0, [(64, 32), (128, 128), (512, 32)]),
    (workloads.STEFAN, 0, [(1024, 4), (4096, 4), (1024, 16), (8, 2)]),
    (workloads.STEFAN, 1, [(1024, 4), (2048, 16), (4096, 8)])])
def test_an_sm_holds_its_share_of_fp64_tiles_and_no_more(plans, problem, flow, sizes):
    """Two FP64 blocks on an SM take twice as long: shared memory (228 KB an SM, 1 KB
    of it reserved per block, about 0.2 KB of static arrays in the kernel) admits
    ceil(tiles / 152) blocks."""
    for size in sizes:
        solo = plans("fp64", problem, flow, [size])[1]
        share = -(-solo["tiles"] // 152)
        assert solo["t"] >= 2 and solo["smem"] <= 230400
        assert share * (solo["smem"] + 1024 + 256) <= 228 * 1024 < (share + 1) * (solo["smem"] + 1024), size


def band_cost(plan, nx, ny, n):
    """(waves, waves x the rows a band computes) of n lattices on 152 SMs."""
    pairs, threads = (nx + 1) // 2, plan["threads"]
    s = max(1, pairs // threads)
    while -(-pairs // s) + min(s - 1, 2) > threads:
        s += 1
    bands = -(-ny // plan["rows"])
    waves = -(-n * s * bands // (152 * (12 // (threads // 32))))
    return waves, waves * (-(-ny // bands) + 2)


@pytest.mark.parametrize("prec,size,n,most", [
    ("fp32", (256, 128), 256, 90), ("bf16sr", (256, 128), 256, 90), ("bf16sr", (128, 64), 512, 50),
    ("fp32", (128, 64), 512, 50), ("fp16", (256, 128), 230, 90)])
def test_bands_of_many_members_fill_their_waves(plans, prec, size, n, most):
    """One band per member left 44 % of a wave empty (a cost of 130 for 256 x 128, 66
    for 128 x 64)."""
    batch = plans(prec, workloads.CAVITY, 1, [size] * n)[0]
    assert batch["threads"] > 0 and band_cost(batch, *size, n)[1] <= most


@pytest.mark.parametrize("nx,ny", [(2048, 1024), (1024, 1024), (1500, 700), (700, 500), (3000, 3000), (16, 65535), (5000, 200),
                                   (4500, 2), (8192, 64)])
def test_bands_of_one_lattice_take_one_wave(plans, nx, ny):
    solo = plans("fp32", workloads.CAVITY, 1, [(nx, ny)])[1]
    assert solo["threads"] > 0 and 1 <= solo["rows"] and band_cost(solo, nx, ny, 1)[0] == 1


@pytest.mark.parametrize("nx,ny,bands", [(65536, 8, False), (65536, 16, False), (131072, 8, False), (65536, 4, True),
                                         (131072, 4, True), (131072, 16, True), (32768, 16, True), (262144, 2, True)])
def test_wide_lattices_of_few_rows(plans, nx, ny, bands):
    assert (plans("fp32", workloads.CAVITY, 1, [(nx, ny)])[1]["threads"] > 0) == bands


@pytest.mark.parametrize("prec,size,n,solo_pf,batch_pf", [
    ("bf16sr", (2048, 1024), 1, 0, 4), ("fp16", (2048, 1536), 1, 32, 4), ("fp16", (4096, 4096), 1, 32, 4),
    ("bf16", (256, 128), 48, 0, 0), ("fp16sr", (256, 128), 64, 0, 4), ("fp32", (2048, 1024), 2, 0, 0)])
def test_16_bit_storage_beyond_l2_prefetches(plans, prec, size, n, solo_pf, batch_pf):
    solo = plans(prec, workloads.CAVITY, 1, [size] * n)[1]
    assert solo["batch_prefetch"] == batch_pf
    if prec != "fp32":
        assert solo["prefetch16"] == solo_pf


@pytest.mark.parametrize("prec,problem,flow,n,rows,prefetch", [
    ("fp32", workloads.CAVITY, 1, 32, 2, 0), ("bf16sr", workloads.CAVITY, 1, 32, 3, 0), ("bf16sr", workloads.CAVITY, 1, 64, 3, 4),
    ("fp32", workloads.STEFAN, 0, 16, 2, 0), ("fp32", workloads.STEFAN, 0, 32, 3, 0), ("fp32", workloads.CAVITY, 0, 64, 3, 0),
    ("fp32", workloads.STEFAN, 1, 16, 2, 0), ("fp32", workloads.STEFAN, 1, 32, 2, 4),
    ("fp16", workloads.STEFAN, 0, 4, 3, 0), ("fp16", workloads.STEFAN, 1, 16, 4, 0), ("bf16", workloads.CAVITY, 0, 16, 3, 0),
    ("bf16", workloads.CAVITY, 0, 32, 4, 0), ("bf16", workloads.CAVITY, 0, 64, 4, 4)])
def test_batch_shapes(plans, prec, problem, flow, n, rows, prefetch):
    """Rows per block and prefetch distance by storage, problem and total size."""
    solo = plans(prec, problem, flow, [(256, 128)] * n)[1]
    assert (solo["batch_rows"], solo["batch_prefetch"]) == (rows, prefetch)


@pytest.mark.parametrize("prec,size,n", [("fp32", (64, 32), 2), ("fp32", (2048, 1024), 2), ("bf16sr", (256, 128), 1)])
def test_the_choice_can_be_given_back(plans, prec, size, n):
    solo = plans(prec, workloads.CAVITY, 1, [size] * n)[1]
    assert (solo["one"], solo["batch_one"]) == (0, 0)
    assert (solo["auto"], solo["batch_auto"]) == (1, 1)
