"""Calls of the CUDA runtime that are refused: the library is linked a second time with
stand-ins in front of cudaMalloc that return an error code at a chosen call
and touch no device.  A refused call returns its status, and the next one on the same grid
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
#include <cuda_runtime.h>
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
                   ["-Xlinker", "--wrap=cudaMalloc"], check=True)
    _lib.load()
    keep, _lib._lib = _lib._lib, None
    lib = _lib.load(so)
    lib.fake_malloc.argtypes, lib.fake_malloc.restype = [C.c_long], None
    lib.fake_seen.restype = C.c_long
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
        if path.startswith("precond"):
            return torch.equal(a, b)
        return (a - b).abs().max().item() <= 1e-6 * (b - st.t_amb).abs().max().item()

    call, refused = PATHS[path], 0
    g = ThermalGrid.from_stack(nx, ny, st)
    ref = call(g, st, P, r)
    g.close()
    for k in range(200):
        g = ThermalGrid.from_stack(nx, ny, st)
        faked.fake_malloc(k)
        try:
            assert same(call(g, st, P, r), ref), k
        except ThermalError as e:
            assert e.status == 2, (k, e)
            refused += 1
        n = faked.fake_seen()
        faked.fake_malloc(-1)
        assert same(call(g, st, P, r), ref), k
        torch.cuda.synchronize()
        g.close()
        if n <= k:
            break
    assert n <= k and refused >= 15, (n, refused)
