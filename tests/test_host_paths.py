"""The library's host code without a GPU: its sources linked against a CUDA runtime that counts calls and fails the ones it is told
to (tests/fake_cudart.cpp).  Covers what a working GPU does not show: which route a call takes when the driver refuses something."""
import ctypes as C
import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

from paper_2608_14624_b200 import binding as cs
from paper_2608_14624_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
OUT_OF_MEMORY = 2
DEVICE_MEMORY, HOST_MEMORY = 2, 1            # cudaMemoryType
WORKSPACE, BUF = 1 << 40, 1 << 41            # addresses nobody follows


@pytest.fixture(scope="module")
def host_library(tmp_path_factory):
    """The library's sources linked against the counting runtime; returns the path."""
    out = tmp_path_factory.mktemp("host_paths")
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcicc", "-O0", "-Xptxas", "-O0",
             "-I", os.path.join(build.ROOT, "include")]
    nvcc = os.environ.get("NVCC", "nvcc")

    def compile_one(src):
        obj = str(out / (os.path.basename(src) + ".o"))
        subprocess.run([nvcc, *flags, "-c", "-o", obj, src], check=True, capture_output=True)
        return obj

    with ThreadPoolExecutor(8) as pool:
        objs = list(pool.map(compile_one, build.sources() + [os.path.join(HERE, "fake_cudart.cpp")]))
    so = str(out / "libcachescout_host.so")
    subprocess.run([nvcc, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", so, *objs], check=True, capture_output=True)
    return so


@pytest.fixture
def rt(host_library, tmp_path):
    """A fresh copy of that library (what it has learnt about a device is kept per process), as the binding's own for one test."""
    so = str(shutil.copy(host_library, tmp_path))
    saved = cs._lib, cs.LIB_PATH
    cs._lib, cs.LIB_PATH = None, so
    L = cs.lib()
    L.fake_calls.argtypes, L.fake_fail.argtypes = [C.c_char_p], [C.c_char_p, C.c_int, C.c_int, C.c_int]
    yield L
    cs._lib, cs.LIB_PATH = saved


def calls(rt, name):
    return rt.fake_calls(name.encode())


def make_ctx(rt, **kw):
    p, ctx = cs.make_params(**kw), C.c_void_p()
    assert rt.cs_create(C.byref(p), WORKSPACE, cs.cs_workspace_bytes(p), None, C.byref(ctx)) == cs.CS_OK
    return ctx.value


def index(n):
    return cs.cs_block_index(n, BUF, BUF, BUF, BUF, BUF, None, None)


@pytest.mark.parametrize("call,skip", [("cudaGraphCreate", 0), ("cudaGraphAddNode", 0), ("cudaGraphAddNode", 7), ("cudaGraphInstantiate", 0),
                                       ("cudaGraphExecNodeSetParams", 0), ("cudaGraphExecNodeSetParams", 11), ("cudaGraphLaunch", 0),
                                       ("cudaGraphLaunch", 2), ("cudaThreadExchangeStreamCaptureMode", 0), ("cudaStreamIsCapturing", 1)])
def test_selects_are_launched_one_by_one_when_their_graph_fails(rt, call, skip):
    """Two lists of a large index, five times.  Whatever the driver refuses of their graph, at whichever call: the call succeeds by
    single launches, no error is left behind, and a graph that failed is not tried again."""
    ctx = make_ctx(rt, n_agents=12, n_chains=4, max_blocks=400_000)
    cs.cs_set_select_path(ctx, cs.CS_SELECT_MULTI)
    idx = index(300_000)
    rt.fake_fail(call.encode(), skip, 1, OUT_OF_MEMORY)
    by_graph = []
    for _ in range(5):
        launched, graphs, n0 = calls(rt, "cs_sel_"), calls(rt, "cudaGraphLaunch"), cs.cs_launch_count(ctx)
        cs.cs_select_step(ctx, idx, 5, 100, 100, BUF, BUF, None, None, BUF, BUF, stream=0)
        assert cs.cs_launch_count(ctx) - n0 == 12
        single = calls(rt, "cs_sel_") - launched
        assert single in (0, 12)
        assert single == 12 or calls(rt, "cudaGraphLaunch") == graphs + 1
        by_graph.append(single == 0)
        assert rt.cs_last_cuda_error(ctx) == 0 and rt.cudaGetLastError() == 0
    if call == "cudaStreamIsCapturing":
        assert by_graph == [False, False, True, True, True]          # (not the graph's fault: the next call builds it)
    elif (call, skip) == ("cudaGraphLaunch", 2):
        assert by_graph == [False, True, True, False, False]
    else:
        assert not any(by_graph)
    cs.cs_destroy(ctx)
    assert calls(rt, "cudaGraphCreate") - (call == "cudaGraphCreate") == calls(rt, "cudaGraphDestroy")


def select_kernels(rt):
    """(cluster, whole-GPU, chain) select launches so far."""
    return tuple(sum(calls(rt, name) for name in names) for names in (("cs_select_cluster_kernel", "cs_select_step_kernel"), ("cs_select_grid_kernel",), ("cs_sel_",)))


CLUSTER, GRID, CHAIN = (1, 0, 0), (0, 1, 0), (0, 0, 6)


@pytest.mark.parametrize("path", [cs.CS_SELECT_AUTO, cs.CS_SELECT_CLUSTER, cs.CS_SELECT_MULTI])
@pytest.mark.parametrize("n,k,later", [(65_536, 4_000, CLUSTER), (65_537, 2_047, CLUSTER), (65_537, 2_048, GRID), (131_072, 100, CLUSTER), (131_073, 100, GRID),
                                       (262_144, 200_000, GRID), (262_145, 100, GRID), (262_145, 50_000, GRID), (262_145, 50_001, CHAIN), (1 << 25, 100, GRID),
                                       ((1 << 25) + 1, 100, CHAIN)])
def test_route_of_a_select(rt, n, k, later, path):
    """Which kernels a list takes on its first call and from the second one on, on both sides of every line; a captured first call counts as a later one."""
    first = CLUSTER if n <= 262_144 else CHAIN
    if path != cs.CS_SELECT_AUTO:
        first = later = first if path == cs.CS_SELECT_CLUSTER else CHAIN
    for captured in (0, 1):
        ctx = make_ctx(rt, n_agents=12, n_chains=4, max_blocks=n + 100)
        cs.cs_set_select_path(ctx, path)
        for call in range(4):
            rt.fake_capturing(captured and call == 0)
            before, n0 = select_kernels(rt), cs.cs_launch_count(ctx)
            if call < 3:
                cs.cs_select_victims(ctx, index(n), 5, 1, k, BUF, BUF, stream=0)
            else:                                               # (a list that has not been asked for)
                cs.cs_select_prefetch(ctx, index(n), 5, k, BUF, BUF, stream=0)
            took = tuple(b - a for a, b in zip(before, select_kernels(rt)))
            assert took == (later if call in (1, 2) or (captured and call == 0) else first), (captured, call)
            assert cs.cs_launch_count(ctx) - n0 == sum(took)
        cs.cs_destroy(ctx)


@pytest.mark.parametrize("n,lists,instead", [(200_000, 1, CLUSTER), (200_000, 3, CLUSTER), (300_000, 1, CHAIN), (300_000, 3, (0, 0, 18))])
@pytest.mark.parametrize("call,skip", [("launch", 0), ("cudaFuncSetAttribute", 0), ("cudaFuncSetAttribute", 4)])
def test_a_refused_whole_gpu_select_goes_the_other_way(rt, n, lists, instead, call, skip):
    """The driver refuses the launch or its shared memory: the call succeeds by the cluster or the chain, no error is left behind, and later calls do not
    ask again."""
    ctx = make_ctx(rt, n_agents=12, n_chains=4, max_blocks=400_000)
    select = lambda: (cs.cs_select_step(ctx, index(n), 5, 100, 100, BUF, BUF, BUF, BUF, BUF, BUF, stream=0) if lists == 3 else
                      cs.cs_select_victims(ctx, index(n), 5, 0, 100, BUF, BUF, stream=0))
    select()
    rt.fake_fail(call.encode(), skip, 1, OUT_OF_MEMORY)
    for _ in range(3):
        before, graphs, n0 = select_kernels(rt), calls(rt, "cudaGraphLaunch"), cs.cs_launch_count(ctx)
        select()
        took = tuple(b - a for a, b in zip(before, select_kernels(rt)))
        assert took == instead or (calls(rt, "cudaGraphLaunch") == graphs + 1 and took == (0, 0, 0) and instead[2] == 18)
        assert cs.cs_launch_count(ctx) - n0 == sum(instead)
        assert rt.cs_last_cuda_error(ctx) == 0 and rt.cudaGetLastError() == 0
    cs.cs_destroy(ctx)


@pytest.mark.parametrize("device,kind,odd,by_kernel", [(0, DEVICE_MEMORY, 0, 8), (1, DEVICE_MEMORY, 0, 0), (0, HOST_MEMORY, 0, 0),
                                                       (0, 0, 0, 0), (0, DEVICE_MEMORY, 1, 0)])
def test_model_is_exported_by_a_kernel_to_its_own_gpu_only(rt, device, kind, odd, by_kernel):
    """The export kernel stores to memory of the context's GPU; another GPU's memory, host memory, memory unknown to the runtime and odd
    addresses are copied by the runtime, one copy per table."""
    ctx = make_ctx(rt, n_agents=12, n_chains=4)
    rt.fake_pointers(device, kind)
    copies = calls(rt, "cudaMemcpyAsync")
    cs.cs_get_model(ctx, *[BUF + 4096 * i + odd for i in range(8)], stream=0)
    assert calls(rt, "cs_export_kernel") == (1 if by_kernel else 0)
    assert calls(rt, "cudaMemcpyAsync") - copies == 8 - by_kernel
    cs.cs_destroy(ctx)


@pytest.mark.parametrize("call,code", [("cudaOccupancyMaxActiveClusters", OUT_OF_MEMORY), ("cudaFuncSetAttribute", OUT_OF_MEMORY), (None, 0)])
@pytest.mark.parametrize("A,kernel", [(12, "cs_refresh_kernelILi1"), (64, "cs_refresh_wide_kernel"), (256, "cs_refresh_wide_kernel"),
                                      (300, "cs_refresh_wide_kernel")])
def test_the_learner_runs_where_no_cluster_size_can_be_found(rt, call, code, A, kernel):
    """When the driver does not say that any cluster fits (an error, or none), the refresh takes a kernel that needs none and a long
    batch one CTA; every call succeeds and leaves no error."""
    if call:
        rt.fake_fail(call.encode(), 0, -1, code)
    else:
        rt.fake_clusters(0)
    ctx = make_ctx(rt, n_agents=A, n_chains=4)
    for n in (3, 2000):
        before = calls(rt, kernel)
        cs.cs_observe_invocations(ctx, BUF, BUF, None, n, stream=0)
        assert calls(rt, kernel) == before + 1
    assert calls(rt, "cs_observe_kernel") == 1 and calls(rt, "cs_refresh_kernelILi8") == 0
    assert rt.cs_last_cuda_error(ctx) == 0 and rt.cudaGetLastError() == 0
    cs.cs_destroy(ctx)
