"""FP64 products by exact digit arithmetic (csrc/fp64_digits.cu) against the
DFMA tile classes on the same environment: H_eff*psi from prepared images and
from operands cut in the kernel, the adjoint's one-off lists (every operand
orientation and identity factor), graded, zero, huge and non-finite vectors.

Both evaluate the same sums in FP64 accuracy.  A sum of n terms by FP64 FMAs
is within n 2^-53 of its terms' magnitudes; the lists here have at most a few
thousand products of at most 100 x 100 terms, whose errors add up like random
ones, so 1e-13 of the result's norm (900 units of 2^-53) bounds the distance of
two such evaluations with a wide margin and is far below any digit lost (2^-48).
"""
import os

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2305_05581_gb300 import Context, DEFAULT_LIB, TNS_FP64  # noqa: E402
from paper_2305_05581_gb300.autograd import arena_tensor  # noqa: E402

TOL = 1e-13
# sectors of 1 to 16, 17 to 32, around 64 and above (ragged), off-centre (wide blocks), edge steps
CASES = [(5, 5, 1, 8, 0, 0), (8, 8, 0, 256, 3, 0), (10, 9, 1, 90, 7, 0), (11, 11, 1, 130, 5, 5),
         (12, 12, 0, 130, 5, 2), (13, 13, 1, 260, 6, 3), (13, 13, 1, 260, 4, 3)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(DEFAULT_LIB):
        from paper_2305_05581_gb300 import build as b
        b.build()


def _ctx(kernel, system):
    N, n, s2, D, k, ms = system
    h, v = synth.integrals(N, 3.0, 60 + N + k)
    bonds, sites = synth.random_mps(N, n, s2, D, center=k, seed=k, max_sectors=ms)
    if kernel:
        os.environ["TNS_FP64_KERNEL"] = kernel
    try:
        ctx = Context(device=0, stream=torch.cuda.current_stream().cuda_stream)
    finally:
        os.environ.pop("TNS_FP64_KERNEL", None)
    ctx.load_integrals(h, v)
    ctx.mps_import(N, n, s2, D, bonds, sites)
    ctx.build_env(k)
    return ctx, k, ctx.psi_layout(k)


def _vector(kind, desc, length, nvec):
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(nvec, length, device="cuda", dtype=torch.float64, generator=g)
    for i, row in enumerate(desc):
        m, n, off = (int(v) for v in row[6:9])
        blk = x[:, off:off + m * n].view(nvec, m, n)
        if kind == "graded":  # rows and columns over six decades each, blocks over 60
            blk *= 10.0 ** (-6 * torch.rand(m, 1, device="cuda", dtype=torch.float64, generator=g))
            blk *= 10.0 ** (-6 * torch.rand(1, n, device="cuda", dtype=torch.float64, generator=g) - 60 * (i % 2))
        elif kind == "sparse":  # zero rows, zero columns, zero blocks
            blk[:, ::2] = 0.0
            blk[:, :, 1::3] = 0.0
            if i % 3 == 0:
                blk.zero_()
        elif kind == "huge" and i % 4 == 0:  # beyond what the fixed-point form holds
            blk *= 1e120
    return x


def _apply(ctx, k, x):
    y = torch.empty_like(x)
    ctx.heff_apply_ptr(k, x.data_ptr(), y.data_ptr(), x.shape[0], TNS_FP64)
    torch.cuda.synchronize()
    return y


def _close(a, b):
    return float(torch.linalg.norm(a - b)) <= TOL * float(torch.linalg.norm(b))


@pytest.mark.parametrize("system", CASES)
@pytest.mark.parametrize("kind", ["normal", "graded", "sparse", "huge"])
def test_heff_matches_dfma(system, kind):
    dg, k, (desc, length) = _ctx(None, system)
    ref, _, _ = _ctx("dfma", system)
    for nvec in (1, 3):  # three vectors: their images grow
        x = _vector(kind, desc, length, nvec)
        assert _close(_apply(dg, k, x), _apply(ref, k, x))
    assert torch.equal(_apply(dg, k, x[:1]), _apply(dg, k, x)[:1])


@pytest.mark.parametrize("system", CASES[2:])
def test_heff_without_images_matches_dfma(system):
    """A device budget with no room for images: operands cut in the kernel."""
    ref, _, _ = _ctx("dfma", system)
    dg, k, (desc, length) = _ctx("digits", system)
    x = _vector("graded", desc, length, 2)
    want = _apply(ref, k, x)
    dg.set_memory_budget(dg.memory_stats()["device_used"] + (1 << 26))
    try:
        assert _close(_apply(dg, k, x), want)
    finally:
        dg.set_memory_budget(0)


@pytest.mark.parametrize("system", CASES)
def test_adjoint_matches_dfma(system):
    out = []
    for kernel in (None, "dfma"):
        ctx, k, (desc, length) = _ctx(kernel, system)
        x, yb = _vector("graded", desc, length, 1)[0], _vector("normal", desc, length, 1)[0]
        res = [torch.zeros(length, device="cuda", dtype=torch.float64)]
        res += [torch.zeros_like(arena_tensor(ctx, k, side)) for side in (0, 1)]
        ctx.heff_adjoint_ptr(k, x.data_ptr(), yb.data_ptr(), *(r.data_ptr() for r in res))
        torch.cuda.synchronize()
        out.append(res)
    for a, b in zip(*out):
        assert _close(a, b)


@pytest.mark.parametrize("system", [CASES[1], CASES[3]])
def test_adjoint_lists_kept_for_the_step(system):
    """The adjoint's lists outlive a call: other vectors, a subset of the
    gradients and an arena changed before build_env give what a context that
    never ran it before gives (both FP64, so within the bound above)."""
    ctx, k, (desc, length) = _ctx(None, system)
    ref, _, _ = _ctx("dfma", system)
    arenas = [arena_tensor(c, k, 0) for c in (ctx, ref)]

    def grads(c, x, yb, which):
        res = [torch.zeros(length, device="cuda", dtype=torch.float64)]
        res += [torch.zeros_like(arena_tensor(c, k, side)) for side in (0, 1)]
        c.heff_adjoint_ptr(k, x.data_ptr(), yb.data_ptr(), *(r.data_ptr() if w else 0 for r, w in zip(res, which)))
        torch.cuda.synchronize()
        return res

    a, b = _vector("normal", desc, length, 2)
    for x, yb, which in ((a, b, (1, 1, 1)), (b, a, (1, 1, 1)), (a + b, b, (0, 1, 0)), (a, a - b, (1, 0, 1))):
        for g, w in zip(grads(ctx, x, yb, which), grads(ref, x, yb, which)):
            assert _close(g, w)
    for arena, c in zip(arenas, (ctx, ref)):
        arena.mul_(0.5)
        c.build_env(k)
    for g, w in zip(grads(ctx, a, b, (1, 1, 1)), grads(ref, a, b, (1, 1, 1))):
        assert _close(g, w)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_entries_reach_the_same_outputs(bad):
    system = CASES[3]
    dg, k, (desc, length) = _ctx(None, system)
    ref, _, _ = _ctx("dfma", system)
    x = _vector("normal", desc, length, 1)
    x[0, length // 2] = bad
    a, b = _apply(dg, k, x), _apply(ref, k, x)
    fine = torch.isfinite(b)
    assert not bool(fine.all())
    assert torch.equal(torch.isfinite(a), fine) and torch.equal(torch.isnan(a), torch.isnan(b))
    assert _close(a[fine], b[fine])
    y = _apply(dg, k, _vector("normal", desc, length, 1))  # and nothing of it stays
    assert bool(torch.isfinite(y).all())
