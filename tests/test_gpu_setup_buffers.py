"""Buffers that a solver keeps from one preconditioner setup to the next."""
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from tests.helpers import ROOT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsv():
    from tests.helpers import build_library
    build_library()
    import paper_1602_05901_gb300 as m
    return m


def _apply(torch, s, r):
    z = torch.full_like(r, float("nan"))
    s.apply(r, z)
    torch.cuda.synchronize()
    return z


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_coarsening_changes_on_one_solver(rsv, precision):
    """Both pressure hierarchies of a grid of at most gmg_max_coarse cells have one geometric level, but only the geometric
    one keeps that level's dense inverse: setups in turn on one solver give the same bits as on a solver of their own."""
    torch = pytest.importorskip("torch")
    p = synth.make_problem(9, 8, 6, seed=31)
    A = rsv.Matrix(p.nx, p.ny, p.nz)
    A.set_values(p.vals)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    r = torch.from_numpy(np.random.default_rng(32).standard_normal(p.n)).cuda().to(dtype)
    setups = {"amg": dict(coarsening="amg", gmg_max_levels=8, gmg_max_coarse=64), "gmg": {}}
    alone = {}
    for name, kw in setups.items():
        s = rsv.Solver(A, precision=precision)
        s.setup("cpr", **kw)
        alone[name] = _apply(torch, s, r)
    s = rsv.Solver(A, precision=precision)
    for name in ("amg", "gmg", "amg", "gmg"):
        s.setup("cpr", **setups[name])
        assert torch.equal(_apply(torch, s, r), alone[name]), name


# cudaMalloc that reports no memory at its n-th call from now (n = rsv_test_fail_at, 0: never).
FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
int rsv_test_fail_at = 0;
int cudaMalloc(void **p, size_t bytes) {
    static int (*real)(void **, size_t) = 0;
    if (!real) real = (int (*)(void **, size_t))dlsym(dlopen("libcudart.so.13", RTLD_LAZY), "cudaMalloc");
    if (rsv_test_fail_at > 0 && --rsv_test_fail_at == 0) return 2;
    return real(p, bytes);
}
"""

CHILD = r"""
import ctypes
import numpy as np
import torch
import paper_1602_05901_gb300 as rsv
import synth
fail_at = ctypes.c_int.in_dll(ctypes.CDLL(None), "rsv_test_fail_at")
p = synth.make_problem(13, 11, 9, seed=33)
A = rsv.Matrix(p.nx, p.ny, p.nz)
A.set_values(p.vals)
r0 = torch.from_numpy(np.random.default_rng(34).standard_normal(p.n)).cuda()
for precision, dtype in (("fp64", torch.float64), ("mixed", torch.float32)):
    r = r0.to(dtype)

    def apply(s):
        z = torch.full_like(r, float("nan"))
        s.apply(r, z)
        torch.cuda.synchronize()
        return z

    s = rsv.Solver(A, precision=precision)
    s.setup("cpr")
    ref = apply(s)
    for n in range(1, 200):
        s = rsv.Solver(A, precision=precision)
        fail_at.value = n
        try:
            s.setup("cpr")
        except rsv.RsvError as e:
            assert e.status in (rsv.RSV_ENOMEM, rsv.RSV_ECUDA), (n, e.status)
        else:
            assert fail_at.value > 0, n
            break
        assert fail_at.value == 0, n
        s.setup("cpr")
        assert torch.equal(apply(s), ref), n
    fail_at.value = 0
    assert n > 20, n
print("ok")
"""


def test_setup_after_a_failed_allocation(rsv, tmp_path):
    """Each device allocation of a CPR setup fails in turn (a fake cudaMalloc; no memory is exhausted): the setup reports it,
    and the next one on the same solver works and gives the same bits as on a new one."""
    pytest.importorskip("torch")
    src, lib = tmp_path / "fake.c", tmp_path / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib))
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stdout + out.stderr
