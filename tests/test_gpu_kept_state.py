"""State that outlives a call: row parts on digit products, and the adjoint's lists
across a two-site step and another site.
"""
import os

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2305_05581_gb300 import Context, DEFAULT_LIB, TNS_FP64  # noqa: E402
from paper_2305_05581_gb300.autograd import arena_tensor  # noqa: E402

# two FP64 evaluations of a few thousand products of up to 100 x 100 terms, of the result's norm
TOL = 1e-13


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(DEFAULT_LIB):
        from paper_2305_05581_gb300 import build as b
        b.build()


def _ctx(kernel, N, n, s2, D, k, ms):
    h, v = synth.integrals(N, 3.0, 7)
    bonds, sites = synth.random_mps(N, n, s2, D, center=k, seed=k, max_sectors=ms)
    os.environ.update(TNS_FP64_KERNEL=kernel, TNS_AUTOTUNE="0")  # one schedule: equal runs are equal bit for bit
    try:
        ctx = Context(device=0, stream=torch.cuda.current_stream().cuda_stream)
    finally:
        os.environ.pop("TNS_FP64_KERNEL")
        os.environ.pop("TNS_AUTOTUNE")
    ctx.load_integrals(h, v)
    ctx.mps_import(N, n, s2, D, bonds, sites)
    ctx.build_env(k)
    return ctx


def _randn(*shape):
    g = torch.Generator(device="cuda").manual_seed(9)
    return torch.randn(*shape, device="cuda", dtype=torch.float64, generator=g)


def _close(a, b):
    return float(torch.linalg.norm(a - b)) <= TOL * float(torch.linalg.norm(b))


@pytest.mark.parametrize("nparts", [1, 3])
def test_row_parts_on_digits(nparts):
    system = (13, 13, 1, 260, 6, 3)
    k = system[4]
    ctx, ref = _ctx("digits", *system), _ctx("dfma", *system)
    _, length = ctx.psi_layout(k)
    x = _randn(2, length)
    total = torch.zeros_like(x)
    for part in range(nparts):
        ys = []
        for c in (ctx, ref):
            y = torch.empty_like(x)
            for _ in range(2):
                c.heff_apply_part_ptr(k, x.data_ptr(), y.data_ptr(), part, nparts, 2, TNS_FP64)
            torch.cuda.synchronize()
            ys.append(y)
        assert _close(*ys)
        total += ys[0]
    y = torch.empty_like(x)
    ref.heff_apply_ptr(k, x.data_ptr(), y.data_ptr(), 2, TNS_FP64)
    torch.cuda.synchronize()
    assert _close(total, y)


def test_adjoint_across_a_step_and_another_site():
    """A context that took the gradients at this site before gives those of one that never did after a step has changed
    the site tensors, at the next site, and back."""
    system = (10, 10, 0, 60, 4, 0)
    k = system[4]

    def grads(ctx, site):
        _, length = ctx.psi_layout(site)
        x, yb = _randn(2, length)
        res = [torch.zeros(length, device="cuda", dtype=torch.float64)]
        res += [torch.zeros_like(arena_tensor(ctx, site, side)) for side in (0, 1)]
        ctx.heff_adjoint_ptr(site, x.data_ptr(), yb.data_ptr(), *(r.data_ptr() for r in res))
        torch.cuda.synchronize()
        return res

    def step(ctx, site, right):
        _, length = ctx.psi_layout(site)
        x0 = _randn(length).cpu()
        ctx.step(site, right, system[3], tol=1e-9, max_iter=200, precision=TNS_FP64, x0_host_ptr=x0.data_ptr())

    out = []
    for before in (True, False):
        ctx = _ctx("dfma", *system)
        seen = []
        if before:
            grads(ctx, k)
            grads(ctx, k)
        step(ctx, k, True)
        for site in (k + 1, k):
            ctx.build_env(site)
            seen.append(grads(ctx, site))
            seen.append(grads(ctx, site))
        out.append(seen)
        ctx.close()
    for a, b in zip(*out):
        for u, w in zip(a, b):
            assert torch.equal(u, w) and float(w.abs().max()) > 0
