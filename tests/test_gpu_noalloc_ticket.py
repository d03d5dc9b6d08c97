"""hca_o2_residual_noalloc counts its blocks' arrivals in scratch memory that
calls share.  Calls that overlapped (the caller must serialise them) may leave
a count behind; the calls after them must not take it for their own arrivals.
Any count up to the most blocks a call has is left, then lattices of other
chunk counts and other fields follow, twice each; all must agree with the
oracle (tolerance as in the entry point's other tests)."""

import ctypes
import os
import subprocess

import pytest

from gpu_helpers import random_states
from oracle import params as Pm
from paper_2105_00448_gb300 import _build, hca
from test_zz_no_alloc import device_arrays, oracle_rel_residual

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SHAPES = [(30, 41, 33), (20, 30, 64), (3, 5, 40), (1, 1, 7)]   # 410, 600, 15 and 1 chunks


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("noalloc") / "libnoalloc_ticket.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-shared", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-I", _build.INCLUDE, "-I", _build.CSRC,
                    os.path.join(HERE, "cuda", "noalloc_ticket.cu"), "-o", out], check=True, capture_output=True, text=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("left", [0, 1, 14, 15, 409, 410, 599, 600, 2048])
def test_a_left_over_count_is_not_taken_for_arrivals(lib, left, rng):
    cases = []
    for nz, ny, nx in SHAPES:
        st = random_states((nz, ny, nx), rng)
        st.reshape(-1)[0] = Pm.VESSEL
        K_prev = rng.uniform(0.0, 20.0, st.shape)
        for _ in range(2):
            K = rng.uniform(0.0, 20.0, st.shape)
            ref, tol = oracle_rel_residual(st, K_prev, K, Pm.Config(nx=nx, ny=ny, nz=nz))
            cases.append((hca.make_config(nx, ny, nz), device_arrays(st, K_prev, K), ref, tol))
    assert lib.noalloc_add_arrivals(left) == 0
    for cfg, args, ref, tol in cases + cases[::-1]:
        got = ctypes.c_double()
        assert lib.hca_o2_residual_noalloc(ctypes.byref(cfg), *[ctypes.c_void_p(a.data_ptr()) for a in args],
                                           ctypes.byref(got), None) == 0
        assert abs(got.value - ref) <= tol
