"""What the host side launches, without a GPU: the library's objects linked with a stand-in for the CUDA runtime."""
import ctypes as C
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def objects(tmp_path_factory):
    from paper_2609_34606_b200 import build
    out = tmp_path_factory.mktemp("fake")
    nvcc = build.nvcc_path()

    def compile_one(src):
        obj = out / (src + ".o")
        # (no GPU code is run: the kernels are left unoptimised, which takes seconds)
        subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-Xcicc", "-O0", "-std=c++17", "-Xcompiler", "-fPIC",
                        "-c", "-o", str(obj), os.path.join(build.CSRC, src)], check=True, capture_output=True)
        return str(obj)

    with ThreadPoolExecutor(8) as pool:
        objs = list(pool.map(compile_one, build.SOURCES))
    fake = out / "fake.o"
    subprocess.run([nvcc, "-std=c++17", "-Xcompiler", "-fPIC", "-c", "-o", str(fake), os.path.join(HERE, "fake_cuda_runtime.cpp")],
                   check=True, capture_output=True)
    return objs + [str(fake)], out


@pytest.fixture
def lib(objects, request):
    """A copy of the library of its own, so that nothing is kept from one test to the next."""
    objs, out = objects
    path = out / (request.node.name.replace("[", "_").replace("]", "") + ".so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", str(path)] + objs, check=True, capture_output=True)
    return C.CDLL(str(path))


class Context:
    """A context over made-up device addresses, with `n` tokens appended."""

    def __init__(self, lib, H, d, max_pages, max_topk, max_q=4680, n=0, flags=0, lin_mode=0):
        from paper_2609_34606_b200 import hsa
        self.lib, self.H, self.d, self.max_topk = lib, H, d, max_topk
        cfg = hsa.hsa_config(H, d, 64, max_pages, max_q, max_topk, lin_mode, 0, 0.0, flags)
        bufs = hsa.hsa_buffers(0x10000000, 0x20000000, 0x30000000, 0x40000000)
        self.ctx = C.c_void_p()
        assert lib.hsa_create(C.byref(self.ctx), C.byref(cfg), C.byref(bufs), None) == 0
        while n > 0:
            m = min(n, max_q)
            assert lib.hsa_append_kv(self.ctx, C.c_void_p(0x1000), C.c_void_p(0x2000), m, C.c_int64(H * d), C.c_int64(d), None) == 0
            n -= m

    def q_args(self, n_q):
        return self.ctx, C.c_void_p(0x1000), n_q, C.c_int64(self.H * self.d), C.c_int64(self.d), C.c_int64(1 << 40), 0

    def select(self, n_q=256, group=0):
        return self.lib.hsa_select_blocks(*self.q_args(n_q), C.c_void_p(0x3000), group, C.c_void_p(0x4000), C.c_void_p(0x5000), None)

    def select_adaptive(self, n_q=256):
        return self.lib.hsa_select_blocks_adaptive(*self.q_args(n_q), C.c_float(0.35), C.c_float(1.0), 0, C.c_void_p(0x4000),
                                                   C.c_void_p(0x5000), None, None)

    def forward(self, n_q, stream=0, group=0):
        none = C.c_void_p(None)
        return self.lib.hsa_forward(*self.q_args(n_q), C.c_void_p(0x4000), C.c_void_p(0x5000), group, none, none, C.c_int64(0),
                                    C.c_int64(0), C.c_int64(0), C.c_void_p(0x6000), C.c_int64(self.H * self.d), C.c_int64(self.d),
                                    0, C.c_void_p(stream))


def launches(lib):
    out = []
    for i in range(lib.fake_launches()):
        name, grid, smem = C.create_string_buffer(400), (C.c_int * 3)(), C.c_longlong()
        dev = lib.fake_launch(i, name, 400, grid, C.byref(smem))
        out.append((name.value.decode(), tuple(grid), smem.value, dev))
    return out


@pytest.mark.parametrize("d,n_blocks,adaptive", [(128, 1700, True), (128, 1800, True), (64, 6144, True), (128, 5000, False),
                                                 (128, 6144, False)])
def test_selection_on_every_device_of_a_process(lib, d, n_blocks, adaptive):
    """Each device gets its own shared-memory limit for the selection kernels, whichever came first."""
    for dev in (0, 1, 0, 2):
        lib.fake_set_device(dev)
        ctx = Context(lib, 4, d, n_blocks, n_blocks, n=n_blocks * 64, flags=2)
        for n_q in (256, 4680):
            lib.fake_reset()
            assert (ctx.select_adaptive(n_q) if adaptive else ctx.select(n_q)) == 0
            names = [l[0] for l in launches(lib)]
            assert names and all(l[3] == dev for l in launches(lib)) and "select_cluster" in names[-1]


@pytest.mark.parametrize("kernel,group,flags", [("topk_kernel", 128, 0), ("select_fused", 0, 4), ("select_fused", 128, 4)])
def test_selections_of_two_threads_keep_each_others_shared_memory(lib, kernel, group, flags):
    """A selection over a shorter history that another thread issues between the shared-memory limit and the launch
    of one over a longer history does not lower the limit under it."""
    long, short = (Context(lib, 2, 128, n, 64, n=n * 64, flags=flags) for n in (50000, 11000))
    results = []
    other = C.CFUNCTYPE(None)(lambda: results.append(short.select(256, group)))
    lib.fake_reset()
    lib.fake_on_smem_limit(other)
    assert long.select(256, group) == 0 and results == [0]
    used = [l[2] for l in launches(lib) if kernel in l[0]]
    assert used == [11000 * 4, 50000 * 4]


@pytest.mark.parametrize("H,tiles,alone,sums", [
    (2, 5, 0, False), (2, 6, 0, True), (12, 6, 0, True), (12, 7, 0, False), (12, 7, 1, True), (12, 8, 0, False), (12, 9, 0, True),
    (16, 6, 0, False), (16, 8, 0, True), (20, 8, 0, False), (20, 8, 1, False), (20, 10, 0, True), (24, 9, 1, True), (40, 5, 1, False)])
def test_causal_sums_where_they_pay(lib, H, tiles, alone, sums):
    """Which causal chunks make sums over page groups: by query tiles, heads and whether a sparse branch follows; the products run
    in the instance that goes with it."""
    n = tiles * 128 - 5
    ctx = Context(lib, H, 128, 80, 32, max_q=n, n=n, flags=1, lin_mode=1)
    none, ts = C.c_void_p(None), C.c_int64(H * 128)
    lib.fake_reset()
    assert lib.hsa_forward(ctx.ctx, C.c_void_p(0x1000), n, ts, C.c_int64(128), C.c_int64(0), 1, C.c_void_p(0x4000), C.c_void_p(0x5000), 0,
                           none, none, C.c_int64(0), C.c_int64(0), C.c_int64(0), C.c_void_p(0x6000), ts, C.c_int64(128),
                           2 if alone else 0, none) == 0
    names = [l[0] for l in launches(lib)]
    assert sum("chunk_sums_kernel" in x for x in names) == sums
    assert sum("causal_linear_kernelILi128ELb%d" % sums in x for x in names) == 1


def test_forwards_of_short_lists_share_no_scratch(lib):
    """Two forwards of one context may run at the same time if their lists are short: they are not split through
    the workspace, which holds nothing for that, and take the same route on every stream and under capture."""
    workspace, cluster, plain = ("hsa_forward_kernelILi128ELi%dE" % i for i in (1, 2, 0))

    def kernel(ctx, n_q, stream=0):
        lib.fake_reset()
        assert ctx.forward(n_q, stream) == 0
        (name, grid, _, _), = launches(lib)
        return next(k for k in (workspace, cluster, plain) if k in name), grid

    ctx = Context(lib, 2, 128, 130, 128, n=130 * 64)
    routes = [kernel(ctx, 256, s) for s in (0, 0x70, 0)]
    lib.fake_set_capturing(0x70, 1)
    routes.append(kernel(ctx, 256, 0x70))
    assert set(routes) == {(cluster, (2 * 8, 2, 1))}
    assert kernel(ctx, 4680) == (plain, (37, 2, 1))
    assert kernel(Context(lib, 2, 128, 20, 20, n=20 * 64), 256)[0] == plain      # never long enough
    assert kernel(Context(lib, 2, 128, 300, 300, n=300 * 64), 256)[0] == workspace
    from paper_2609_34606_b200 import hsa
    sizes = {hsa.hsa_query_sizes(hsa.hsa_config(2, 128, 64, 300, 4680, k, 1, 0, 0.0, 0)).workspace for k in (1, 47, 48, 256)}
    assert len(sizes) == 1
