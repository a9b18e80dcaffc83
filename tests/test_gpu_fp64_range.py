"""FP64 products hold entry by entry and for every magnitude, as an FMA chain does.

H_eff*psi and its adjoint on vectors whose states carry weights over many
decades, and on vectors and operators near the small end of the FP64 range.

Entries: on a basis of determinants and with density-density integrals alone
(h_ii and (ii|jj)) every operator that counts is diagonal, so that weakly weighted
states get their result from weakly weighted entries and nothing larger hides its
error; with all integrals their sums have larger terms too.  Each entry is held
against its own sum S = sum |L| |X| |R|^T (the oracle's heff_apply_abs).  A sum
of n terms by FMAs is within n 2^-53 S, and its roundings add up like random
ones; the lists here have at most some 4,000 products, sqrt(4000) 2^-53 = 2^-47,
so two such evaluations are within 2^-45 S.

Magnitudes: without an underflow every FP64 operation commutes with powers of
two, so the product of 2^-p x is compared with 2^-p times the product of x.
"""
import os

import numpy as np
import pytest

import synth
import test_gpu_fp64_digits
from oracle import dmrg as O3

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2305_05581_gb300 import Context, DEFAULT_LIB, TNS_FP64, blocks_to_vector, vector_to_blocks  # noqa: E402
from paper_2305_05581_gb300.autograd import arena_tensor  # noqa: E402

TOL_ENTRY = 2.0 ** -45
TOL = 1e-13  # of the result's norm: two FP64 evaluations of a few thousand products of up to 100 x 100 terms


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(DEFAULT_LIB):
        from paper_2305_05581_gb300 import build as b
        b.build()


def _ctx(kernel, N, n, s2, D, k, h, v, bonds, sites):
    if kernel:
        os.environ["TNS_FP64_KERNEL"] = kernel
    try:
        ctx = Context(device=0, stream=torch.cuda.current_stream().cuda_stream)
    finally:
        os.environ.pop("TNS_FP64_KERNEL", None)
    ctx.load_integrals(h, v)
    ctx.mps_import(N, n, s2, D, bonds, sites)
    ctx.build_env(k)
    return ctx


def _determinants(N, n, s2, k):
    """A random MPS with the blocks beside the step replaced by 0/1 isometries: every left and right state is one
    determinant."""
    bonds, sites = synth.random_mps(N, n, s2, 10 ** 6, center=k, seed=1)
    for b in range(N):
        left, right = dict(bonds[b]), dict(bonds[b + 1])
        if b < k:
            for qr, dr in bonds[b + 1]:
                keys = [((qr[0] - a, qr[1] - c), s) for s, (a, c) in enumerate(synth.SITE_QN)]
                at = 0
                for key in keys:
                    if key[0] in left:
                        sites[b][key] = np.ascontiguousarray(np.eye(dr)[at:at + left[key[0]]])
                        at += left[key[0]]
                assert at == dr
        elif b > k + 1:
            for ql, dl in bonds[b]:
                at = 0
                for s, (a, c) in enumerate(synth.SITE_QN):
                    qr = (ql[0] + a, ql[1] + c)
                    if qr in right:
                        sites[b][(ql, s)] = np.ascontiguousarray(np.eye(dl)[:, at:at + right[qr]])
                        at += right[qr]
                assert at == dl
    return bonds, sites


@pytest.fixture(scope="module", params=[(8, 8, 0, 3, True), (10, 9, 1, 4, True), (8, 8, 0, 3, False)],
                ids=["N8_density", "N10_density", "N8"])
def determinants(request):
    N, n, s2, k, density = request.param
    h, v = synth.integrals(N, 3.0, 5)
    if density:
        i = np.arange(N)
        keep = np.zeros_like(v)
        keep[i[:, None], i[:, None], i[None], i[None]] = 1.0
        h, v = np.diag(np.diag(h)), v * keep
    bonds, sites = _determinants(N, n, s2, k)
    heff = O3.DenseHeff(O3.Integrals(h, v), bonds, sites, k, n, s2)
    yield (N, n, s2, 10 ** 6, k, h, v, bonds, sites), heff, synth.psi_keys(bonds, N, n, s2, k)


def _graded(keys, decades):
    """Gaussian blocks whose left and right states carry weights over that many decades each."""
    rng = np.random.default_rng(11)
    wl, wr, out = {}, {}, {}
    for key, (m, n) in keys:
        wl.setdefault(key[0], 10.0 ** (-decades * rng.random(m)))
        wr.setdefault(key[3], 10.0 ** (-decades * rng.random(n)))
        out[key] = rng.standard_normal((m, n)) * wl[key[0]][:, None] * wr[key[3]][None]
    return out


def _apply(ctx, k, x):
    y = torch.empty_like(x)
    ctx.heff_apply_ptr(k, x.data_ptr(), y.data_ptr(), x.shape[0], TNS_FP64)
    torch.cuda.synchronize()
    return y


def _entries_hold(desc, got, want, bound):
    got, want = vector_to_blocks(desc, got), vector_to_blocks(desc, want)
    for q in bound:
        err = np.abs(got[q] - want[q])
        assert np.all(err <= TOL_ENTRY * bound[q]), (q, float(np.max(err / np.maximum(bound[q], 1e-300))))


# the FP64 kernels by the library's rule, and digits wherever a list has images: pieces without a certificate, all of
# them in some of these systems, are then done again by the FMA kernel
KERNELS = pytest.mark.parametrize("kernel", [None, "digits"])


@KERNELS
@pytest.mark.parametrize("decades", [0, 4, 9])
def test_entries_of_weak_states(determinants, decades, kernel):
    system, heff, keys = determinants
    k = system[4]
    X = _graded(keys, decades)
    bound = heff.apply_abs(X)
    ctx, ref = _ctx(kernel, *system), _ctx("dfma", *system)
    desc, length = ctx.psi_layout(k)
    x = torch.tensor(blocks_to_vector(desc, length, X), device="cuda")[None]
    got, want = _apply(ctx, k, x), _apply(ref, k, x)
    _entries_hold(desc, got[0].cpu().numpy(), want[0].cpu().numpy(), bound)
    _entries_hold(desc, want[0].cpu().numpy(), blocks_to_vector(desc, length, heff.apply(X)), bound)


@pytest.mark.parametrize("decades", [4, 9])
def test_entries_of_the_adjoint(determinants, decades):
    """Xbar = H_eff Ybar for a symmetric H_eff, so the same sums bound it."""
    system, heff, keys = determinants
    k = system[4]
    Y = _graded(keys, decades)
    ctx, ref = _ctx(None, *system), _ctx("dfma", *system)
    desc, length = ctx.psi_layout(k)
    x = torch.tensor(blocks_to_vector(desc, length, _graded(keys, 0)), device="cuda")
    yb = torch.tensor(blocks_to_vector(desc, length, Y), device="cuda")
    out = []
    for c in (ctx, ref):
        xb = torch.zeros_like(x)
        c.heff_adjoint_ptr(k, x.data_ptr(), yb.data_ptr(), xb.data_ptr(), 0, 0)
        torch.cuda.synchronize()
        out.append(xb.cpu().numpy())
    _entries_hold(desc, out[0], out[1], heff.apply_abs(Y))


SYSTEMS = [(8, 8, 0, 256, 3, 0), (13, 13, 1, 260, 6, 3)]


def _random(system):
    N, n, s2, D, k, ms = system
    h, v = synth.integrals(N, 3.0, 60 + N)
    bonds, sites = synth.random_mps(N, n, s2, D, center=k, seed=k, max_sectors=ms)
    return (N, n, s2, D, k, h, v, bonds, sites)


def _close(a, b):
    return float(torch.linalg.norm(a - b)) <= TOL * float(torch.linalg.norm(b))


UP = 2.0 ** 400  # brings results back where their norms do not underflow


def _small(desc, x, p, part):
    """2^-p x; with part > 1 only one block in `part`, and the others at 2^-(p - 40)."""
    x = x.clone()
    for i, row in enumerate(desc):
        m, n, off = (int(v) for v in row[6:9])
        x[:, off:off + m * n] *= 2.0 ** -(p if i % part == 0 else p - 40)
    return x


MAGNITUDES = pytest.mark.parametrize("p,part", [(430, 1), (714, 1), (764, 1), (960, 1), (764, 4), (960, 4)])


@pytest.mark.parametrize("system", SYSTEMS)
@MAGNITUDES
def test_small_vectors_in_the_adjoint(system, p, part):
    args = _random(system)
    k = args[4]
    grads = []
    for kernel in (None, "dfma"):
        c = _ctx(kernel, *args)
        desc, length = c.psi_layout(k)
        g = torch.Generator(device="cuda").manual_seed(7)
        x = torch.randn(1, length, device="cuda", dtype=torch.float64, generator=g)
        small = _small(desc, x, p, part)
        res = [torch.zeros(length, device="cuda", dtype=torch.float64)]
        res += [torch.zeros_like(arena_tensor(c, k, side)) for side in (0, 1)]
        c.heff_adjoint_ptr(k, x.data_ptr(), small.data_ptr(), *(r.data_ptr() for r in res))
        torch.cuda.synchronize()
        assert all(float(r.abs().max()) > 0 for r in res)
        grads.append(res)
    for u, w in zip(*grads):
        assert _close(u * UP, w * UP)


@KERNELS
@pytest.mark.parametrize("system", SYSTEMS)
@MAGNITUDES
def test_small_vectors(system, p, part, kernel):
    args = _random(system)
    k = args[4]
    ctx, ref = _ctx(kernel, *args), _ctx("dfma", *args)
    desc, length = ctx.psi_layout(k)
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(1, length, device="cuda", dtype=torch.float64, generator=g)
    small = _small(desc, x, p, part)
    got = _apply(ctx, k, small)
    assert _close(got * UP, _apply(ref, k, small) * UP)
    if part == 1:  # powers of two pass through
        assert _close(got * UP, _apply(ref, k, x) * 2.0 ** (400 - p))


@KERNELS
def test_small_operators_and_small_vector(kernel):
    """Left operators and a vector whose products are near 1e-286: one block of X, and the output blocks of other left
    sectors, which only an operator of the left block reaches."""
    args = _random(SYSTEMS[1])
    k = args[4]
    out = []
    for name in (kernel, "dfma"):
        ctx = _ctx(name, *args)
        desc, length = ctx.psi_layout(k)
        rows = [[int(v) for v in r] for r in desc]
        big = max(rows, key=lambda r: r[6] * r[7])
        g = torch.Generator(device="cuda").manual_seed(7)
        x = torch.zeros(1, length, device="cuda", dtype=torch.float64)
        x[:, big[8]:big[8] + big[6] * big[7]] = 2.0 ** -470 * torch.randn(
            big[6] * big[7], device="cuda", dtype=torch.float64, generator=g)
        arena_tensor(ctx, k, 0).mul_(2.0 ** -480)
        torch.cuda.synchronize()
        ctx.build_env(k)
        y = _apply(ctx, k, x)[0] * 2.0 ** 900
        out.append(torch.cat([y[r[8]:r[8] + r[6] * r[7]] for r in rows if r[:2] != big[:2]]))
    assert float(out[1].abs().max()) > 0
    assert _close(*out)


@pytest.mark.parametrize("system", test_gpu_fp64_digits.CASES)
@pytest.mark.parametrize("kind", ["normal", "graded", "sparse", "huge"])
def test_digits_of_small_lists(system, kind):
    """Lists that the library leaves to the FMA kernel for their size, on the digit kernel."""
    args = _random(system)
    k = args[4]
    ctx, ref = _ctx("digits", *args), _ctx("dfma", *args)
    desc, length = ctx.psi_layout(k)
    for nvec in (1, 3):
        x = test_gpu_fp64_digits._vector(kind, desc, length, nvec)
        assert _close(_apply(ctx, k, x), _apply(ref, k, x))
    assert torch.equal(_apply(ctx, k, x[:1]), _apply(ctx, k, x)[:1])


@pytest.mark.parametrize("graphs", ["0", "1"])
def test_vectors_beyond_the_images(graphs):
    """No memory for the images of more vectors: the call runs on the images there are, with the same results, and the
    one-vector products before and after, by replayed graphs too, stay as they were."""
    args = _random(SYSTEMS[1])
    k = args[4]
    os.environ.update(TNS_GRAPHS=graphs, TNS_AUTOTUNE="0")
    try:
        ctx, free = _ctx(None, *args), _ctx(None, *args)
    finally:
        os.environ.pop("TNS_GRAPHS")
        os.environ.pop("TNS_AUTOTUNE")
    _, length = ctx.psi_layout(k)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(3, length, device="cuda", dtype=torch.float64, generator=g)
    want = _apply(free, k, x)
    one = [_apply(ctx, k, x[:1]) for _ in range(3)]
    ctx.set_memory_budget(ctx.memory_stats()["device_used"] + (1 << 26))
    try:
        assert torch.equal(_apply(ctx, k, x), want)
        one += [_apply(ctx, k, x[:1]) for _ in range(2)]
    finally:
        ctx.set_memory_budget(0)
    assert torch.equal(_apply(ctx, k, x), want)
    one += [_apply(ctx, k, x[:1]) for _ in range(2)]
    assert all(torch.equal(y, want[:1]) for y in one)


def test_first_product_of_a_small_list_allocates_no_images():
    """Below the line by size the first product costs what it costs with the FMA kernel alone."""
    args = _random(SYSTEMS[0])
    k = args[4]
    used = []
    for kernel in (None, "dfma"):
        ctx = _ctx(kernel, *args)
        _, length = ctx.psi_layout(k)
        x = torch.ones(1, length, device="cuda", dtype=torch.float64)
        before = ctx.memory_stats()["device_used"]
        _apply(ctx, k, x)
        used.append(ctx.memory_stats()["device_used"] - before)
        ctx.close()
    assert used[0] == used[1]


@pytest.mark.parametrize("system", SYSTEMS + [(11, 11, 1, 130, 5, 5)])
def test_rounding_has_no_direction(system):
    """Both kernels round to the nearest, so the difference of their results has no component along the result.  The
    entries' errors are a few units of 2^-53 of their typical magnitude and independent, so over n entries the
    component is a few 2^-53 / sqrt(n): 0.05 units at the 5,000 entries of the smallest system.  Dropping the bits
    below the last makes every contribution too small, which shows as 2 to 3.5 units (contributions are larger than
    the results they cancel to), and ties away from zero as 0.17."""
    args = _random(system)
    k = args[4]
    ctx, ref = _ctx("digits", *args), _ctx("dfma", *args)
    _, length = ctx.psi_layout(k)
    assert length > 4000
    g = torch.Generator(device="cuda").manual_seed(3)
    along = []
    for _ in range(8):
        x = torch.randn(1, length, device="cuda", dtype=torch.float64, generator=g)
        got, want = _apply(ctx, k, x), _apply(ref, k, x)
        along.append(float(((got - want) * want).sum() / (want * want).sum()) * 2.0 ** 53)
    assert abs(np.mean(along)) < 0.15, along
