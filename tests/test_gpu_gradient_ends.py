"""The kernels at the two ends of a reverse pass: the outlet flux and the transposed
grad-eps stencil, against float64 sums of the same numbers."""
import numpy as np
import pytest

import oracle as O
from paper_1406_6438_gb300 import workloads as W
from tests._gpu import solver, torch_cuda

pytestmark = pytest.mark.gpu

# (q, (nz, ny, nx)): rows of the outlet plane around the 256 threads and 8 blocks that
# sum it; axes of one and two cells
SHAPES = [(9, (1, 1, 5)), (9, (1, 2, 1)), (9, (1, 255, 4)), (9, (1, 2049, 3)), (9, (1, 5000, 2)),
          (9, (1, 40, 131)), (19, (1, 1, 3)), (19, (2, 3, 2)), (19, (60, 41, 7)), (19, (9, 10, 67))]


def _directions(q):
    r = (-1, 0, 1)
    if q == 9:
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
        dirs = [(x, y, 0) for x in r for y in r]
    else:
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        dirs = [(x, y, z) for x in r for y in r for z in r if abs(x) + abs(y) + abs(z) <= 2]
    return [(e, float(np.float32(w[sum(map(abs, e))]))) for e in dirs]


def _case(q, shape, walls, seed):
    nz, ny, nx = shape
    p = W.params(q=q, nx=nx, ny=ny, nz=nz, wall_mask=walls, tau=0.7, g=(3e-4, 0.0, 0.0),
                 drag_mode=2, k_mode=0, d_p=6.0)
    eps = W.smoothed_noise(shape, 2.0, 0.4, 1.0, seed)
    return p, eps, W.random_state(q, eps, seed + 1, amp=0.02)


@pytest.mark.parametrize("q,shape", SHAPES)
def test_flux_is_the_sum_of_the_outlet(q, shape):
    """Tolerance: eps, rho and u carry an fp32 rounding or two each, relative to the
    cells' magnitudes (the sum itself cancels)."""
    torch = torch_cuda()
    p, eps, f0 = _case(q, shape, 2, seed=sum(shape))
    s = solver(p, eps)
    s.set_populations(torch.from_numpy(f0).cuda())
    J = float(s.flux(shape[2] - 1))
    rho, u = s.moments()
    terms = (eps.reshape(shape).astype(np.float64) * rho.cpu().numpy().reshape(shape) *
             u[0].cpu().numpy().reshape(shape))[:, :, -1]
    assert abs(J - terms.sum()) <= 1e-6 * np.abs(terms).sum()


@pytest.mark.parametrize("walls", [0, 2, 6])
@pytest.mark.parametrize("q,shape", SHAPES)
def test_gradient_stencil(q, shape, walls):
    """lambda = 0, accumulators of 1e4 whose stencil cancels to a difference: to the
    rounding of the result, and 2^-42 of the terms for the two-float sums of 36."""
    torch = torch_cuda()
    if q == 9 and walls == 6:
        pytest.skip("no z walls in two dimensions")
    nz, ny, nx = shape
    D = 2 if q == 9 else 3
    p, eps, _ = _case(q, shape, walls, seed=2)
    s = solver(p, eps)
    rng = np.random.default_rng(5)
    head = (1e4 + rng.standard_normal((1 + D,) + shape)).astype(np.float32)
    head[0] = rng.standard_normal(shape)
    tail = (1e-4 * rng.standard_normal((1 + D,) + shape)).astype(np.float32)
    acc = torch.from_numpy(np.concatenate([head.ravel(), tail.ravel()])).cuda()
    out = s.grad_finalize(s.new_state(), acc).cpu().numpy().reshape(shape)
    G = head.astype(np.float64) + tail
    v = G[0].copy()
    z, y, x = np.meshgrid(*(np.arange(n) for n in shape), indexing="ij")
    for e, w in _directions(q):
        def past(sign):
            yy, zz = y + sign * e[1], z + sign * e[2]
            return ((walls & 2 != 0) & ((yy < 0) | (yy >= ny))) | ((walls & 4 != 0) & ((zz < 0) | (zz >= nz)))
        src = G[:, (z - e[2]) % nz, (y - e[1]) % ny, (x - e[0]) % nx]
        for field, where in ((src, ~past(-1)), (G, past(1))):
            v += np.where(where, 3 * w * sum(e[c] * field[1 + c] for c in range(D)), 0.0)
    assert np.all(np.abs(out - v) <= 2.0 ** -23 * np.abs(v) + 2.0 ** -42 * 1e4 * 36)


def _stencil64(q, shape, walls, lam, G):
    """G_eps + sum w lambda + the transposed stencil in 64 bits; lam[i]: plane i of the
    lambda state, G: the accumulators' sums."""
    e, w, opp = O.lattice(q)[:3]
    w = np.asarray(w, dtype=np.float32).astype(np.float64)
    nz, ny, nx = shape
    z, y, x = np.meshgrid(*(np.arange(n) for n in shape), indexing="ij")
    v = G[0].astype(np.float64)
    for i, ei in enumerate(np.asarray(e)):
        ei = list(ei) + [0] * (3 - len(ei))

        def past(sign):
            yy, zz = y + sign * ei[1], z + sign * ei[2]
            return ((walls & 2 != 0) & ((yy < 0) | (yy >= ny))) | ((walls & 4 != 0) & ((zz < 0) | (zz >= nz)))

        def src(f):
            return f[..., (z - ei[2]) % nz, (y - ei[1]) % ny, (x - ei[0]) % nx]
        v += w[i] * np.where(past(-1), lam[opp[i]], src(lam[i]))
        for field, where in ((src(G), ~past(-1)), (G, past(1))):
            v += np.where(where, 3 * w[i] * sum(ei[c] * field[1 + c] for c in range(len(G) - 1) if ei[c]), 0.0)
    return v


def _finalize(q, shape, walls, lam, acc, bits=32):
    torch = torch_cuda()
    p, eps, _ = _case(q, shape, walls, seed=2)
    s = solver(p, eps)
    s.set_adjoint_precision(bits)
    rows, off = shape[0] * shape[1], 8 if q == 9 else 32
    pitch = s.state_floats // (q * rows) // 32 * 32           # (the state's end is padded too)
    state = s.new_state()
    lam = np.concatenate([lam[..., -1:], lam, lam[..., :1]], axis=-1).reshape(q, rows, -1)   # halo columns
    state[:q * rows * pitch].view(q, rows, pitch)[:, :, off - 1:off + shape[2] + 1] = torch.from_numpy(lam).cuda()
    return s.grad_finalize(state, torch.from_numpy(acc.ravel()).cuda()).cpu().numpy().reshape(shape)


def _cancelling(q, shape, rng, noise):
    """lambda of 1e4 whose weighted sum cancels to about `noise`."""
    lam = np.empty((q,) + shape)
    w0 = float(np.float32(4 / 9 if q == 9 else 1 / 3))
    lam[0] = 1e4
    lam[1:] = -1e4 * w0 / (1 - w0)
    return (lam + noise * rng.standard_normal((q,) + shape)).astype(np.float32)


@pytest.mark.parametrize("walls", [0, 2, 6])
@pytest.mark.parametrize("q,shape", SHAPES)
def test_lambda_and_stencil_cancel(q, shape, walls):
    """lambda of 1e4 whose weighted sums cancel, against a stencil that cancels too: half
    an ulp of the result, and 2^-42 of the terms for the two-float sums of 55."""
    if q == 9 and walls == 6:
        pytest.skip("no z walls in two dimensions")
    rng, D = np.random.default_rng(6), 2 if q == 9 else 3
    lam = _cancelling(q, shape, rng, 1.0)
    head = (1e4 + rng.standard_normal((1 + D,) + shape)).astype(np.float32)
    head[0] = rng.standard_normal(shape)
    tail = (1e-4 * rng.standard_normal((1 + D,) + shape)).astype(np.float32)
    out = _finalize(q, shape, walls, lam, np.stack([head, tail]))
    v = _stencil64(q, shape, walls, lam.astype(np.float64), head.astype(np.float64) + tail)
    assert np.all(np.abs(out - v) <= 2.0 ** -24 * np.abs(v) + 2.0 ** -42 * 1e4 * 55)


@pytest.mark.parametrize("walls", [0, 2, 6])
@pytest.mark.parametrize("q,shape", [(9, (1, 40, 131)), (19, (9, 10, 67))])
def test_64_bit_sums_where_they_are_asked_for(q, shape, walls):
    """set_adjoint_precision(64): terms of at most 20 bits on a grid of 2^-6, so that every
    product with a weight (24 bits) and every sum of 55 of them is exact in 64 bits,
    cancelling to 1e-3: the result is the exact sum rounded once."""
    if q == 9 and walls == 6:
        pytest.skip("no z walls in two dimensions")
    rng, D = np.random.default_rng(7), 2 if q == 9 else 3
    grid = lambda a: (np.round(a * 64) / 64).astype(np.float32)  # noqa: E731
    lam = grid(_cancelling(q, shape, rng, 0.1))
    acc = np.zeros((2, 1 + D) + shape, dtype=np.float32)
    acc[0, 1:] = grid(1e4 + rng.standard_normal((D,) + shape))
    G = acc.astype(np.float64).sum(0)
    G[0] = 0
    acc[0, 0] = -grid(_stencil64(q, shape, walls, lam.astype(np.float64), G))
    G[0] = acc[0, 0]
    v = _stencil64(q, shape, walls, lam.astype(np.float64), G)
    out = _finalize(q, shape, walls, lam, acc, bits=64)
    assert np.all(np.abs(out - v) <= 2.0 ** -24 * np.abs(v))


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("q,shape", [(9, (1, 6, 9)), (19, (4, 5, 6))])
def test_sums_that_leave_the_range_of_floats(q, shape, bits):
    """An infinite or NaN accumulator or lambda gives what a sum in 64 bits gives, and terms
    whose partial sums pass the largest float do not."""
    D = 2 if q == 9 else 3
    for kind in ("inf", "-inf", "nan", "large"):
        lam = np.zeros((q,) + shape, dtype=np.float32)
        acc = np.zeros((2, 1 + D) + shape, dtype=np.float32)
        if kind == "large":
            lam[:] = np.where(np.arange(q) % 2, 3e38, -3e38).reshape((q,) + (1,) * 3)
            acc[0, 1:] = 3e38 * np.sign(np.arange(acc[0, 1:].size) % 3 - 1.0).reshape(acc[0, 1:].shape)
        else:
            acc[0, 0, 0, 2, 3] = acc[0, 1, 0, 4, 4] = float(kind)
            lam[3, 0, 1, 1] = float(kind)
        with np.errstate(invalid="ignore", over="ignore"):
            G = acc.astype(np.float64).sum(0)
            v = _stencil64(q, shape, 2, lam.astype(np.float64), G).astype(np.float32)
        out = _finalize(q, shape, 2, lam, acc, bits)
        assert np.array_equal(np.isnan(out), np.isnan(v)), kind
        ok = ~np.isnan(v)
        assert np.allclose(out[ok], v[ok], rtol=1e-5, atol=1e-30), kind


@pytest.mark.parametrize("q,shape", [(9, (1, 256, 3)), (9, (1, 257, 3)), (19, (16, 16, 3)), (19, (17, 16, 3))])
def test_flux_of_one_block_and_of_a_cluster(q, shape):
    """At the most rows that one block sums and one row more."""
    test_flux_is_the_sum_of_the_outlet(q, shape)
