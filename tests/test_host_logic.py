"""The library's host code on a runtime without a GPU (fake_cudart.cpp): at the limits of device memory, with
memory of another device, and which kernel a call is given.  Kernels do nothing there, so only statuses,
allocations, copies and the names of the kernels count."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gpu_util import MMA_PHASES

HERE = os.path.dirname(os.path.abspath(__file__))
FP16, BF16 = 2, 3
DIMS = (8, 8, 8, 4)
V = 8 * 8 * 8 * 4


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1409_1510_gb300 import build
    build.build()
    objects = [os.path.join(build.BUILD, os.path.basename(f)[:-3] + ".o") for f in build.sources()]
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    out = str(tmp_path_factory.mktemp("fake") / "libhisq_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.cpp")] + objects + ["-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.fake_used.restype = ctypes.c_size_t
    lib.fake_refused.restype = ctypes.c_ulong
    lib.fake_budget.argtypes = [ctypes.c_size_t]
    lib.fake_foreign.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    lib.fake_time.argtypes = [ctypes.c_char_p, ctypes.c_float]
    lib.fake_launched.argtypes = [ctypes.c_char_p]
    lib.fake_copied.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.hisq_residual.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double] + [ctypes.c_void_p] * 3 + [
        ctypes.c_int, ctypes.c_void_p]
    lib.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    return lib


@pytest.fixture
def ctx(fake):
    fake.fake_budget(ctypes.c_size_t(-1).value)
    fake.fake_foreign(None, 0)
    assert fake.hisq_init((ctypes.c_int * 4)(*DIMS), 0, None) == 0
    yield fake
    fake.fake_budget(ctypes.c_size_t(-1).value)
    fake.fake_foreign(None, 0)
    fake.fake_clear_times()
    assert fake.hisq_finalize() == 0


def _device(lib, nbytes):
    p = ctypes.c_void_p()
    assert lib.cudaMalloc(ctypes.byref(p), nbytes) == 0
    return p.value


def _links(lib, canon, naik, prec, recon=18):
    h = ctypes.c_void_p()
    return lib.hisq_links_create(ctypes.byref(h), ctypes.c_void_p(canon), naik, prec, recon), h


@pytest.mark.parametrize("prec", [FP16, BF16])
def test_links_fit_without_their_optional_copy(ctx, prec):
    """Memory for the stored, FP64 and double-single records but not for the tensor-core copy too: the handle
    is created, without that copy."""
    canon = _device(ctx, 4 * V * 18 * 8)
    before = ctx.fake_used()
    rc, h = _links(ctx, canon, 0, prec)
    assert rc == 0
    whole = ctx.fake_used() - before
    copy = V * 18 * 16  # as large as the 16-bit records: 8 links of 36 bytes per site
    assert ctx.hisq_links_destroy(h) == 0 and ctx.fake_used() == before
    for short in (1, copy // 2, copy):
        ctx.fake_budget(before + whole - short)
        rc, h = _links(ctx, canon, 0, prec)
        assert rc == 0, short
        assert ctx.fake_used() - before == whole - copy
        assert ctx.hisq_links_destroy(h) == 0 and ctx.fake_used() == before
    ctx.fake_budget(before + whole - copy - 1)
    rc, h = _links(ctx, canon, 0, prec)
    assert rc != 0 and ctx.fake_used() == before


@pytest.fixture
def residual_buffers(ctx):
    """(context, call, rhs, x, r): FP16 links and device buffers of hisq_residual for two right-hand sides."""
    canon = _device(ctx, 4 * V * 18 * 8)
    handles = [_links(ctx, canon, naik, FP16) for naik in (0, 1)]
    assert [rc for rc, _ in handles] == [0, 0]
    size = 2 * (V // 2) * 48
    bufs = [_device(ctx, size + 4096) for _ in range(3)]

    def call(rhs, x, r):
        ctx.fake_clear()
        assert ctx.hisq_residual(handles[0][1], handles[1][1], 0.1, rhs, x, r, 2, None) == 0
        return [bool(ctx.fake_copied(rhs, 1)), bool(ctx.fake_copied(x, 1)), bool(ctx.fake_copied(r, 0))]

    yield ctx, call, size, bufs
    for p in bufs + [canon]:
        ctx.cudaFree(ctypes.c_void_p(p))


def test_residual_copies_buffers_of_another_device(residual_buffers):
    """The kernels take buffers of the context's device as they are; those of another device, and host
    memory, are copied."""
    ctx, call, size, bufs = residual_buffers
    assert call(*bufs) == [False, False, False]
    for i, p in enumerate(bufs):
        ctx.fake_foreign(p, size)
        assert call(*bufs) == [j == i for j in range(3)]
    ctx.fake_foreign(None, 0)
    host = np.zeros((3, size), np.uint8)
    assert call(*[host[i].ctypes.data for i in range(3)]) == [True, True, True]


def test_residual_stages_an_output_that_overlaps_an_input(residual_buffers):
    """r over part of rhs or x: written through the scratch, so no input is overwritten while it is read."""
    ctx, call, size, (b, x, r) = residual_buffers
    one = size // 2
    assert call(b, x, r) == [False, False, False]
    for over in (b, x):
        wide = _device(ctx, 3 * one)
        # inputs in the first two thirds, r one right-hand side on; then the other way round; then the same
        for at_in, at_r in ((wide, wide + one), (wide + one, wide), (wide, wide)):
            args = [at_in if over == b else b, at_in if over == x else x, at_r]
            assert call(*args)[2], (over == b, at_in - wide, at_r - wide)
        assert call(wide if over == b else b, wide if over == x else x, r) == [False, False, False]
        ctx.cudaFree(ctypes.c_void_p(wide))
    wide = _device(ctx, 2 * size)
    assert call(wide, x, wide + size) == [False, False, False]  # adjacent, not over one another
    ctx.cudaFree(ctypes.c_void_p(wide))


@pytest.mark.parametrize("R", [1, 2])
def test_launches_the_tensor_cores_cannot_take_keep_the_tuned_shape(ctx, R):
    """Where the tensor-core kernel is the fastest, the decomposed Dslash (which it cannot take) runs the
    fastest of the other shapes, not the default one."""
    lt = 8
    assert ctx.hisq_finalize() == 0
    assert ctx.hisq_init((ctypes.c_int * 4)(8, 8, 8, lt), 0, None) == 0
    canon = _device(ctx, 8 * V * 18 * 8)
    (rc0, fat), (rc1, naik) = (_links(ctx, canon, k, BF16) for k in (0, 1))
    slabs = ctypes.c_void_p()
    assert [rc0, rc1] == [0, 0]
    assert ctx.hisq_slabs_create(ctypes.byref(slabs), ctypes.c_void_p(canon), ctypes.c_void_p(canon), BF16, 2) == 0
    name = b"dslash_kernelILi%dELi18ELi%dELi0ELi2E" % (BF16, R)  # plain, two lanes per site
    ctx.fake_time(name, 0.5)
    ctx.fake_time(b"dslash_mma_kernel", 0.1)
    n, shape = 8, [ctypes.c_int() for _ in range(3)]
    assert ctx.hisq_autotune(fat, naik, n, *[ctypes.byref(v) for v in shape]) == 0
    assert shape[2].value == 32
    vec = _device(ctx, n * 8 ** 3 * lt // 2 * 48)
    ctx.fake_clear()
    assert ctx.hisq_slabs_dslash(slabs, ctypes.c_void_p(vec), ctypes.c_void_p(vec), n, 0, None) == 0
    assert ctx.fake_launched(b"dslash_kernel") == ctx.fake_launched(name) > 0
    assert ctx.hisq_slabs_destroy(slabs) == 0
    for p in (canon, vec):
        ctx.cudaFree(ctypes.c_void_p(p))


def _solve(lib, fat, naik, n, half_volume, **params):
    """hisq_cg_solve of one bundle of n; the status is of no interest (no kernel runs)."""
    from paper_1409_1510_gb300 import hisq
    p = hisq.hisq_solver_params()
    assert lib.hisq_default_solver_params(ctypes.byref(p)) == 0
    p.bundle = n
    for k, v in params.items():
        setattr(p, k, v)
    assert lib.hisq_set_solver_params(ctypes.byref(p)) == 0
    vecs = [np.zeros((half_volume, 6)) for _ in range(2 * n)]
    ptrs = [(ctypes.c_void_p * n)(*[v.ctypes.data for v in half]) for half in (vecs[:n], vecs[n:])]
    lib.fake_clear()
    lib.hisq_cg_solve(fat, naik, *ptrs, n, ctypes.c_double(0.1), ctypes.c_double(1e-10))


@pytest.mark.parametrize("prec,phases", sorted(MMA_PHASES.items()))
def test_persistent_tensor_core_phases_by_bundle_size(ctx, prec, phases):
    """Where the separate Dslash is fastest on the tensor cores, the persistent solve takes its tensor-core
    phases for the bundle sizes that they were measured faster at."""
    canon = _device(ctx, 4 * V * 18 * 8)
    (rc0, fat), (rc1, naik) = (_links(ctx, canon, k, prec) for k in (0, 1))
    assert [rc0, rc1] == [0, 0]
    ctx.fake_time(b"dslash_mma_kernel", 0.1)
    for n in range(1, 17):
        _solve(ctx, fat, naik, n, V // 2, inner_prec=prec, persistent_threads=512)
        assert ctx.fake_launched(b"cg_persistent_kernel") == 1
        assert ctx.fake_launched(b"cg_persistent_kernelILi%dELi16E" % prec) == (n in phases), n
    ctx.cudaFree(ctypes.c_void_p(canon))


def test_training_asks_for_its_optional_activations_once(ctx):
    """Memory for the network's workspace but not for the second set of activations: the calls work without
    it and do not try its allocations again, until the workspace itself is made anew."""
    FP32 = 1
    canon = _device(ctx, 4 * V * 18 * 8)
    (rc0, fat), (rc1, naik) = (_links(ctx, canon, k, FP32) for k in (0, 1))
    pc, loss, grad = ctypes.c_void_p(), ctypes.c_double(), np.zeros(408 * 2)
    assert [rc0, rc1, ctx.hisq_pc_create(ctypes.byref(pc), None)] == [0, 0, 0]
    vec = _device(ctx, 3 * V // 2 * 24)

    def call(K):
        before = ctx.fake_refused()
        assert ctx.hisq_pc_loss_grad(pc, fat, naik, ctypes.c_double(0.1), ctypes.c_void_p(vec), ctypes.c_void_p(vec),
                                     K, ctypes.byref(loss), ctypes.c_void_p(grad.ctypes.data)) == 0
        return ctx.fake_refused() - before

    one = V // 2 * 3 * 4 * 8  # a set of activations is four of these per sample
    for K in (1, 2):
        ctx.fake_budget(ctypes.c_size_t(-1).value)
        assert call(K) == 0  # the whole workspace for K fits
        whole = ctx.fake_used()
        assert ctx.hisq_pc_destroy(pc) == 0 and ctx.hisq_pc_create(ctypes.byref(pc), None) == 0
        ctx.fake_budget(whole - 4 * K * one + 3 * K * one)
        assert [call(K) for _ in range(3)] == [1, 0, 0]
        assert ctx.fake_used() == whole - 4 * K * one
    ctx.fake_budget(ctypes.c_size_t(-1).value)
    assert call(3) == 0 and ctx.fake_used() > whole  # a larger workspace asks again
    assert ctx.hisq_pc_destroy(pc) == 0
    for p in (canon, vec):
        ctx.cudaFree(ctypes.c_void_p(p))
