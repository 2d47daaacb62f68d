"""Which kernels a call on the CUDA-core path launches, and what becomes of a launch that the CUDA runtime refuses.

The library's own launch code is built over a stand-in for the runtime (fake_cuda_runtime.cu) that records the launches
and refuses what a case says; nothing runs on a GPU."""
import ctypes
import itertools
import os
import subprocess

import pytest

from paper_2503_17922_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
SMEM = 227 * 1024                   # what a block may have; a kernel's static words come off the dynamic ones
TOO_LARGE, ILLEGAL = 720, 700       # cudaErrorCooperativeLaunchTooLarge, cudaErrorIllegalAddress
ONE, TWO = "score_fused_simt", "score_stats_simt score_pool_simt"
_device = itertools.count()         # what the library has asked of one device it does not ask again


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    nvcc = build._nvcc()
    try:
        subprocess.check_output([nvcc, "--version"])
    except OSError:
        pytest.skip("no nvcc")
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    # (PTX alone: the device code is never loaded.  The stand-in's functions, not those of a runtime that the process has.)
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-O0", "-Xcicc", "-O0", "-std=c++17",
                           "-Xcompiler", "-fPIC", "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-I", os.path.join(build.ROOT, "include"),
                           "-I", build.CSRC, "-o", so, os.path.join(build.CSRC, "score_simt.cu"),
                           os.path.join(HERE, "fake_cuda_runtime.cu")])
    lib = ctypes.CDLL(so)

    def select(rows=16, head_dim=64, n=600, window=8, f32=True, clusters=16, cooperative_error=0, smem=SMEM - 16, device=None):
        log, pending = ctypes.create_string_buffer(256), ctypes.c_int(0)
        err = lib.fake_select(ctypes.c_int(next(_device) if device is None else device), ctypes.c_size_t(smem), clusters,
                              cooperative_error, int(f32), rows, head_dim, n, window, log, ctypes.c_size_t(256),
                              ctypes.byref(pending))
        return err, log.value.decode(), pending.value
    return select


@pytest.mark.parametrize("case,kernels", [
    (dict(), ONE),
    (dict(clusters=1), TWO),                                   # 600 keys are two clusters
    (dict(clusters=2), ONE),
    (dict(window=12), TWO),                                    # windows straddle tiles
    (dict(rows=129), TWO),
    (dict(rows=128, head_dim=284), ONE),
    (dict(rows=128, head_dim=288), TWO),                       # only the two kernels fit shared memory
    (dict(rows=16, head_dim=684), TWO),
    (dict(n=16 + 8 * 2048, clusters=0), TWO),
    (dict(n=16 + 8 * 2049, clusters=0), TWO + " select_topk"),
])
def test_one_launch_or_two(fake, case, kernels):
    assert fake(**case) == (0, kernels, 0)


@pytest.mark.parametrize("f32", [True, False])
@pytest.mark.parametrize("rows", [16, 32, 64, 128])
def test_a_cooperative_launch_that_is_refused_is_served_by_the_two_kernels(fake, rows, f32):
    """The query may answer for more SMs than the context has: then the launch is refused, and the two kernels, none of whose
    blocks waits for another, take the call.  The refusal is not left behind for the next call to report."""
    assert fake(rows=rows, f32=f32, cooperative_error=TOO_LARGE) == (0, TWO, 0)


def test_other_launch_errors_reach_the_caller(fake):
    err, kernels, _ = fake(cooperative_error=ILLEGAL)
    assert err == ILLEGAL and kernels == ""


def test_a_size_that_does_not_fit_is_remembered(fake):
    device = next(_device)
    for _ in range(2):
        assert fake(rows=128, head_dim=288, device=device) == (0, TWO, 0)
        assert fake(rows=128, head_dim=64, device=device) == (0, ONE, 0)


def test_nothing_that_a_block_may_wait_for_is_taken_ahead_of_the_kernel_in_front():
    """A block that starts while the kernel in front still runs holds its SM's tensor memory from no other block: one of that
    kernel's that waited for it would never end, and this block waits for that kernel.  (Read in the source: the way it fails is a GPU
    that hangs.)"""
    with open(os.path.join(build.CSRC, "score_tc.cu")) as f:
        source = f.read()
    body = source[source.index("score_windows_tc(const __grid_constant__ CUtensorMap tmap"):]
    ahead, behind = body[:body.index("pdl_wait();")], body[body.index("pdl_wait();"):]
    assert "take_wave<" in behind and "tmem_alloc" not in ahead and "take_wave<" not in ahead
    helper = source[source.index("void fetch_ahead("):]
    assert "fetch_ahead<" in ahead and "tmem_alloc" not in helper[:helper.index("score_windows_tc(")]
    assert source.count("tmem_alloc(") == 1


@pytest.fixture(scope="module")
def replays(tmp_path_factory):
    nvcc = build._nvcc()
    try:
        subprocess.check_output([nvcc, "--version"])
    except OSError:
        pytest.skip("no nvcc")
    so = str(tmp_path_factory.mktemp("fake-plan") / "libfakeplan.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-O0", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-cudart", "none", "-Xlinker", "-Bsymbolic", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-o", so,
                           os.path.join(build.CSRC, "group_plan.cu"), os.path.join(HERE, "fake_plan_runtime.cu")])
    lib = ctypes.CDLL(so)

    def run(script, failing=""):
        log = ctypes.create_string_buffer(1024)
        lib.fake_replays(script.encode(), failing.encode(), log, ctypes.c_size_t(1024))
        return [step.strip() for step in log.value.decode().split("|")[:-1]]
    return run


A, B = "score:A gather:A record:A", "score:B gather:B record:B"


@pytest.mark.parametrize("script,failing,steps", [
    ("AA", "", [A, A]),
    ("ABBA", "", [A, "wait:B " + B, B, "wait:A " + A]),      # ordered on the device, never on the host
    ("ABB", "wait:B ", [A, "wait:B -", "wait:B " + B]),                    # a move that fails is made again
    ("ABA", "gather:B ", [A, "wait:B score:B gather:B record:B -", "wait:A " + A]),     # what has been launched stays in the order
    ("ABA", "score:B ", [A, "wait:B score:B -", A]),
    ("A!BAB", "", [A, "graph:B -", A, "wait:B " + B]),                     # refused in a recording, and nothing lost
    ("A1BB0A", "", [A, "wait:B graph:B", "wait:B graph:B", "wait:A graph:A"]),      # another device's stream: as a graph from then on
])
def test_replays_of_a_plan_follow_one_another(replays, script, failing, steps):
    """A replay is put behind the one before it by an event, whatever streams the two are on; the host waits for nothing."""
    assert replays(script, failing) == steps
