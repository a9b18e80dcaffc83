"""The adjoint under a device budget, on the test-only plain-loop build of the
engine: a call needs no more than one side's gradients of the catalogue's and the
partial sums' blocks beside what is there, and keeps nothing where memory is
short; without a budget its lists and buffers stay for the step, with the same
results.
"""
import os
import subprocess

import numpy as np
import pytest

import synth
from paper_2305_05581_gb300.binding import Context, TnsError

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIB = os.path.join(ROOT, "_build", "libtns_hostcheck.so")


@pytest.fixture(scope="module")
def hostlib():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    src = [os.path.join(ROOT, "tests", "hostcheck", "hostcheck.cpp"),
           os.path.join(ROOT, "paper_2305_05581_gb300", "csrc", "engine.cpp")]
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", LIB] + src)
    return LIB


def _adjoint(ctx, k, x, yb):
    res = [np.zeros(x.size)] + [np.zeros(ctx.env_arena(k, side)[1]) for side in (0, 1)]
    ctx.heff_adjoint_ptr(k, x.ctypes.data, yb.ctypes.data, *(r.ctypes.data for r in res))
    return res


@pytest.mark.parametrize("N,n,s2,D,k", [(6, 6, 0, 12, 2), (8, 7, 1, 30, 3)])
def test_adjoint_fits_beside_the_step(hostlib, N, n, s2, D, k):
    h, v = synth.integrals(N, 2.0, 31 + N)
    bonds, sites = synth.random_mps(N, n, s2, D, center=k, seed=k)
    ctx = Context(path=hostlib, prefix="tnshc_")
    ctx.load_integrals(h, v)
    ctx.mps_import(N, n, s2, D, bonds, sites)
    ctx.build_env(k)
    _, length = ctx.psi_layout(k)
    rng = np.random.default_rng(5)
    x, yb = rng.standard_normal(length), rng.standard_normal(length)
    used = ctx.memory_stats()["device_used"]
    want = _adjoint(ctx, k, x, yb)
    kept = ctx.memory_stats()["device_used"] - used
    assert kept > 0  # both sides' buffers and copies of the vectors
    ctx.build_env(k)  # gives them back
    used = ctx.memory_stats()["device_used"]
    both = kept - 2 * 8 * length
    ctx.set_memory_budget(used + both, 0)  # what the gradients take, without copies of the vectors
    for a, b in zip(_adjoint(ctx, k, x, yb), want):
        assert np.array_equal(a, b)
    assert ctx.memory_stats()["device_used"] == used
    ctx.set_memory_budget(used + both // 4, 0)
    with pytest.raises(TnsError):
        _adjoint(ctx, k, x, yb)
    assert ctx.memory_stats()["device_used"] == used
    ctx.set_memory_budget(0, 0)
    for a, b in zip(_adjoint(ctx, k, x, yb), want):
        assert np.array_equal(a, b)
    ctx.close()
