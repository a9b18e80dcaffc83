"""What the library keeps on the device only to run faster -- the digit images of
FP64 products, the work lists of the adjoint -- goes back when a call needs the
room, before any operator catalogue leaves the device, and the results stay what
they are without a budget.
"""
import os

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2305_05581_gb300 import Context, DEFAULT_LIB, TNS_BF16X3, TNS_FP64  # noqa: E402
from paper_2305_05581_gb300.autograd import arena_tensor  # noqa: E402

N, NE, S2, D, K, SECTORS = 20, 20, 0, 400, 9, 8
SLACK = 32 << 20  # less than the split-BF16 images of this step take


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(DEFAULT_LIB):
        from paper_2305_05581_gb300 import build as b
        b.build()


@pytest.fixture(scope="module")
def state():
    h, v = synth.integrals(N, 5.0, 4)
    return (h, v) + synth.random_mps(N, NE, S2, D, center=K, seed=2, max_sectors=SECTORS)


def _ctx(state):
    h, v, bonds, sites = state
    os.environ["TNS_AUTOTUNE"] = "0"
    try:
        ctx = Context(device=0, stream=torch.cuda.current_stream().cuda_stream)
    finally:
        os.environ.pop("TNS_AUTOTUNE")
    ctx.load_integrals(h, v)
    ctx.mps_import(N, NE, S2, D, bonds, sites)
    ctx.build_env(K)
    return ctx, ctx.psi_layout(K)[1]


def _vector(length):
    g = torch.Generator(device="cuda").manual_seed(5)
    return torch.randn(length, device="cuda", dtype=torch.float64, generator=g)


def _apply(ctx, x, precision):
    y = torch.empty_like(x)
    ctx.heff_apply_ptr(K, x.data_ptr(), y.data_ptr(), 1, precision)
    torch.cuda.synchronize()
    return y


def _adjoint(ctx, x, yb):
    res = [torch.zeros_like(x)] + [torch.zeros_like(arena_tensor(ctx, K, side)) for side in (0, 1)]
    ctx.heff_adjoint_ptr(K, x.data_ptr(), yb.data_ptr(), *(r.data_ptr() for r in res))
    torch.cuda.synchronize()
    return res


def _moved(ctx):
    m = ctx.memory_stats()
    return m["staged"], m["dropped"]


def test_digit_images_make_room(state):
    ref, length = _ctx(state)
    x = _vector(length)
    before = ref.memory_stats()["device_used"]
    want = _apply(ref, x, TNS_BF16X3)
    assert ref.memory_stats()["device_used"] - before > SLACK
    ref.close()
    ctx, _ = _ctx(state)
    before = ctx.memory_stats()["device_used"]
    exact = _apply(ctx, x, TNS_FP64)
    images = ctx.memory_stats()["device_used"] - before
    for _ in range(2):  # a graph that reads the images
        assert torch.equal(_apply(ctx, x, TNS_FP64), exact)
    assert images > 4 * SLACK
    moved = _moved(ctx)
    ctx.set_memory_budget(ctx.memory_stats()["device_used"] + SLACK)
    try:
        assert torch.equal(_apply(ctx, x, TNS_BF16X3), want)
        assert _moved(ctx) == moved
        y = _apply(ctx, x, TNS_FP64)
        assert float(torch.linalg.norm(y - exact)) <= 1e-13 * float(torch.linalg.norm(exact))
        assert torch.equal(_apply(ctx, x, TNS_BF16X3), want)
    finally:
        ctx.set_memory_budget(0)
    ctx.close()


def test_adjoint_lists_make_room(state):
    ref, length = _ctx(state)
    x = _vector(length)
    want = _apply(ref, x, TNS_BF16X3)
    ref.close()
    ctx, _ = _ctx(state)
    before = ctx.memory_stats()["device_used"]
    grads = _adjoint(ctx, x, want)
    assert ctx.memory_stats()["device_used"] - before > 4 * SLACK
    moved = _moved(ctx)
    ctx.set_memory_budget(ctx.memory_stats()["device_used"] + SLACK)
    try:
        assert torch.equal(_apply(ctx, x, TNS_BF16X3), want)
        assert _moved(ctx) == moved
    finally:
        ctx.set_memory_budget(0)
    for a, b in zip(_adjoint(ctx, x, want), grads):
        assert torch.equal(a, b)
    ctx.close()


def test_adjoint_where_memory_is_short(state):
    """Made, run and given back one output at a time, the lists give the same gradients."""
    ctx, length = _ctx(state)
    x = _vector(length)
    yb = x.flip(0)
    before = ctx.memory_stats()["device_used"]
    want = _adjoint(ctx, x, yb)
    kept = ctx.memory_stats()["device_used"] - before
    ctx.build_env(K)
    used = ctx.memory_stats()["device_used"]
    ctx.set_memory_budget(used + kept)
    try:
        for a, b in zip(_adjoint(ctx, x, yb), want):
            assert torch.equal(a, b)
        assert ctx.memory_stats()["device_used"] == used
    finally:
        ctx.set_memory_budget(0)
    ctx.close()
