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
        return dict(zip(keys, v[:5])), dict(zip(keys + ("tiles", "smem"), v[5:]))

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
