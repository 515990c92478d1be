"""Calls of the CUDA runtime that are refused: the library is linked a second time with
stand-ins in front of cudaMalloc and the kernel launch that return an error code at a
chosen call and touch no device.  A refused call returns its status, and the next one on the same grid
is right: nothing half-built is used."""
import ctypes as C
import glob
import os
import subprocess

import numpy as np
import pytest

import thermal_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda.h>
#include <cuda_runtime.h>
static int no_coop = 0;  // refuse cooperative launches
static long refused = 0;
extern "C" void fake_no_coop(int on) { no_coop = on; refused = 0; }
extern "C" long fake_refused() { return refused; }
extern "C" cudaError_t __real_cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**);
extern "C" cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
  for (unsigned i = 0; no_coop && i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative) {
      ++refused;
      return cudaErrorCooperativeLaunchTooLarge;
    }
  return __real_cudaLaunchKernelExC(c, f, a);
}
// a stream whose kernels get part of the SMs (at least `want`; *got in fact)
extern "C" int green_stream(unsigned want, void** stream, unsigned* got) {
  CUdevResource all, part;
  unsigned n = 1;
  CUdevResourceDesc desc;
  CUgreenCtx g;
  CUstream s;
  if (cuDeviceGetDevResource(0, &all, CU_DEV_RESOURCE_TYPE_SM)) return 1;
  if (cuDevSmResourceSplitByCount(&part, &n, &all, nullptr, 0, want) || n < 1) return 2;
  if (cuDevResourceGenerateDesc(&desc, &part, 1)) return 3;
  if (cuGreenCtxCreate(&g, desc, 0, CU_GREEN_CTX_DEFAULT_STREAM)) return 4;
  if (cuGreenCtxStreamCreate(&s, g, CU_STREAM_NON_BLOCKING, 0)) return 5;
  *stream = s;
  *got = part.sm.smCount;
  return 0;
}
static long left = -1;   // cudaMalloc calls until the one that is refused, -1: none
static long seen = 0;
extern "C" void fake_malloc(long n) { left = n; seen = 0; }
extern "C" long fake_seen() { return seen; }
extern "C" cudaError_t __real_cudaMalloc(void**, size_t);
extern "C" cudaError_t __wrap_cudaMalloc(void** p, size_t n) {
  ++seen;
  if (left >= 0 && left-- == 0) return cudaErrorMemoryAllocation;
  return __real_cudaMalloc(p, n);
}
"""


@pytest.fixture(scope="module")
def faked(tmp_path_factory):
    """libthermal linked with the stand-ins; the binding uses it for this module's tests."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__ as ge
    from paper_2606_17850_gb300 import _lib, build
    ge.build()
    d = tmp_path_factory.mktemp("refuse")
    (d / "fake.cu").write_text(SRC)
    so = str(d / "libthermal_faked.so")
    objs = sorted(os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build._sources())
    subprocess.run([build.nvcc()] + build.ARCH + ["-Xcompiler", "-fPIC", "-shared", "-o", so, str(d / "fake.cu")] + objs +
                   ["-Xlinker", "--wrap=cudaMalloc", "-Xlinker", "--wrap=cudaLaunchKernelExC", "-lcuda"], check=True)
    _lib.load()
    keep, _lib._lib = _lib._lib, None
    lib = _lib.load(so)
    lib.fake_malloc.argtypes, lib.fake_malloc.restype = [C.c_long], None
    lib.fake_seen.restype = lib.fake_refused.restype = C.c_long
    yield lib
    lib.fake_malloc(-1)
    _lib._lib = keep


def _power(st, nx, ny):
    return torch.from_numpy(ti.power_cells(st, nx, ny, [ti.density_uniform_hotspots(nx, ny, 4)
                                                        for _ in st.power_layers()], np.float32)).cuda()


def _run(g, st, P, o):
    T = torch.full((g.n,), st.t_amb, dtype=torch.float64, device="cuda")
    g.run_transient([P], 2, 5, 1e-4, T, tol_rel=1e-9, **o)
    return T


PATHS = {
    "precond-cheb": lambda g, st, P, r: g.precond(r, 1e-4, precond="cheb", cheb_degree=9),
    "precond-cheb-tiles": lambda g, st, P, r: g.precond(r, 1e-4, precond="cheb", cheb_degree=9, cheb_fuse=4),
    "precond-mg": lambda g, st, P, r: g.precond(r, 0.0, precond="mg"),
    "precond-zline": lambda g, st, P, r: g.precond(r, 0.0, precond="zline"),
    "steady-mg": lambda g, st, P, r: g.solve_steady(P, precond="mg", tol_rel=1e-9)[0],
    "steady-fp64": lambda g, st, P, r: g.solve_steady(P, precision="fp64", cheb_degree=9, tol_rel=1e-9)[0],
    "steady-adaptive": lambda g, st, P, r: g.solve_steady(P, precision="adaptive", cheb_degree=9, tol_rel=1e-9)[0],
    "run-cubic": lambda g, st, P, r: _run(g, st, P, dict(precond="cheb", cheb_degree=9, guess=3)),
}


@pytest.mark.parametrize("path", PATHS)
def test_refused_allocation_leaves_the_grid_usable(faked, path):
    """Every allocation of a first call refused in turn: TH_ENOMEM or the right result, and
    the next call on that grid gives the result of an undisturbed one."""
    from paper_2606_17850_gb300 import ThermalError, ThermalGrid
    nx, ny, st = 68, 41, ti.stack_c2()
    P = _power(st, nx, ny)
    r = torch.from_numpy(ti.random_vector(nx * ny * st.L, 5).astype(np.float32)).cuda()

    def same(a, b):  # solves stop at 1e-9 of ||b||; applications are deterministic
        if path == "precond-cheb":  # on chip, or by chunks: the bound between the forms
            return (a - b).abs().max().item() <= 2.5e-6 * b.abs().max().item()
        if path.startswith("precond"):
            return torch.equal(a, b)
        return (a - b).abs().max().item() <= 1e-6 * (b - st.t_amb).abs().max().item()

    call, refused, absorbed = PATHS[path], 0, 0
    other = torch.cuda.Stream()
    g = ThermalGrid.from_stack(nx, ny, st)
    ref = call(g, st, P, r)
    g.close()
    for k in range(200):
        g = ThermalGrid.from_stack(nx, ny, st)
        faked.fake_malloc(k)
        try:
            assert same(call(g, st, P, r), ref), k
            absorbed += faked.fake_seen() > k
        except ThermalError as e:
            assert e.status == 2, (k, e)
            refused += 1
        n = faked.fake_seen()
        faked.fake_malloc(-1)
        with torch.cuda.stream(other):  # what the failed call left is ready for any stream
            assert same(call(g, st, P, r), ref), k
        torch.cuda.synchronize()
        g.close()
        if n <= k:
            break
    assert n <= k and refused >= 15, (n, refused)
    # only the words of the on-chip solve can be done without
    assert absorbed == (1 if path in ("precond-cheb", "run-cubic") else 0)


FORMS = [(200, 160, "c2", 12), (68, 41, "c1", 9), (131, 37, "c2", 13), (76, 37, "mol", 8)]
STACKS = {"c1": ti.stack_c1, "c2": ti.stack_c2, "mol": ti.stack_mol}


def _calls(g, st, P, r, k, fuse):
    """One application (own buffers, and z = r) and the solves of a first use, as tensors."""
    from paper_2606_17850_gb300 import _lib, api
    o = dict(precond="cheb", cheb_degree=k, cheb_fuse=fuse)
    out = [g.precond(r, 1e-4, **o)]
    z, opts = r.clone(), api.make_opts(**o)
    _lib.check(_lib.load().thermal_precond_apply(g.handle, 1e-4, C.byref(opts), C.c_void_p(z.data_ptr()),
                                                 C.c_void_p(z.data_ptr()),
                                                 C.c_void_p(torch.cuda.current_stream().cuda_stream)))
    out.append(z)
    for graph in (0, 1):
        out.append(g.solve_steady(P, tol_rel=1e-9, use_graph=graph, **o)[0] - st.t_amb)
        out.append(_run(g, st, P, dict(use_graph=graph, guess=1, **o)) - st.t_amb)
    return out


def _agree(a, b, exact):
    for i, (x, y) in enumerate(zip(a, b)):
        if i < 2 and exact:
            assert torch.equal(x, y), i
        else:
            assert (x - y).abs().max().item() <= 1e-6 * y.abs().max().item(), i


@pytest.mark.parametrize("nx,ny,mk,k", FORMS)
def test_refused_cooperative_launch_takes_the_chunks(faked, nx, ny, mk, k):
    """Where the cooperative launch is refused, every call gives what the chunk kernels give
    (one step per launch where nx % 4 != 0), polled and in a graph."""
    from paper_2606_17850_gb300 import ThermalGrid
    st = STACKS[mk]()
    P, r = _power(st, nx, ny), torch.from_numpy(ti.random_vector(nx * ny * st.L, 5).astype(np.float32)).cuda()
    g = ThermalGrid.from_stack(nx, ny, st)
    want = _calls(g, st, P, r, k, 4)
    faked.fake_no_coop(1)
    try:
        got = _calls(g, st, P, r, k, 0)
        assert faked.fake_refused() >= 6
    finally:
        faked.fake_no_coop(0)
    _agree(got, want, True)
    _agree(_calls(g, st, P, r, k, 0), want, False)  # and on chip again
    torch.cuda.synchronize()
    g.close()


def _part_stream(faked):
    ptr, got = C.c_void_p(), C.c_uint()
    if faked.green_stream(16, C.byref(ptr), C.byref(got)) != 0:
        pytest.skip("no green contexts here")
    return ptr, got.value


@pytest.mark.parametrize("nx,ny,mk", [(64, 40, "c1"), (200, 150, "c2"), (131, 77, "mol")])
def test_vcycle_on_part_of_the_device(faked, nx, ny, mk):
    """The V-cycle on a stream with 16 SMs, where a cluster of 16 blocks may have no place:
    the same vector, and the solves' results."""
    from paper_2606_17850_gb300 import ThermalGrid
    ptr, _ = _part_stream(faked)
    st = STACKS[mk]()
    P, r = _power(st, nx, ny), torch.from_numpy(ti.random_vector(nx * ny * st.L, 5).astype(np.float32)).cuda()
    g = ThermalGrid.from_stack(nx, ny, st)

    def calls():
        T = [g.solve_steady(P, precond="mg", tol_rel=1e-9, use_graph=q)[0] - st.t_amb for q in (0, 1)]
        return [g.precond(r, 0.0, precond="mg")] + T

    want = calls()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.ExternalStream(ptr.value)):
        have = calls()
        torch.cuda.synchronize()
    assert torch.equal(have[0], want[0])
    for x, y in zip(have[1:], want[1:]):
        assert (x - y).abs().max().item() <= 1e-6 * y.abs().max().item()
    g.close()


def test_on_chip_tiles_fit_the_streams_part_of_the_device(faked):
    """A stream of a green context with 16 SMs: grids with more tiles run the chunk kernels,
    smaller ones stay on chip."""
    from paper_2606_17850_gb300 import ThermalGrid
    ptr, got = _part_stream(faked)
    sms = faked._Z10stream_smsP11CUstream_st
    sms.argtypes = [C.c_void_p]
    whole = torch.cuda.get_device_properties(0).multi_processor_count
    assert sms(ptr) == got < whole and sms(None) == whole
    part = torch.cuda.ExternalStream(ptr.value)
    for nx, ny, mk, k, fits in ((200, 160, "c2", 12, 0), (288, 201, "c1", 9, 0), (24, 8, "c2", 9, 1), (60, 41, "c1", 12, 1)):
        st = STACKS[mk]()
        P, r = _power(st, nx, ny), torch.from_numpy(ti.random_vector(nx * ny * st.L, 5).astype(np.float32)).cuda()
        torch.cuda.synchronize()
        g = ThermalGrid.from_stack(nx, ny, st)
        want = _calls(g, st, P, r, k, 0 if fits else 4)
        torch.cuda.synchronize()
        with torch.cuda.stream(part):
            have = _calls(g, st, P, r, k, 0)
            torch.cuda.synchronize()
        _agree(have, want, True)
        g.close()
