"""FP64 products on the integer pipe (softfp.h) and the stencils around them.

* The product is correctly rounded: bit-identical to the native one for
  random operands, exact ties, carries into the exponent, powers of 2, zeros
  of both signs and operands near the ends of the normal range.
* A tile takes the integer form only where all its cells lie in [2^-64, 2^64):
  residual and linearisation (F, frozen Jv, material partials through the
  vector-Jacobian product) against the oracle with no, some and all cells
  outside, on whole and ragged tiles.  Tolerance 1e-12 of each cell's term
  scale, as in the parity tests (rounding of a sum of O(10) terms, ~1e-15,
  with a factor 1000 for reordering).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.oracle import Oracle  # noqa: E402
from paper_1302_6303_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def nrd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1302_6303_gb300 import nrd as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_product_bits(nrd):
    rng = np.random.default_rng(3)
    n = 1 << 18
    man = rng.integers(0, 1 << 52, (2, n), dtype=np.uint64)
    # long runs of zeros and ones at either end: ties and carries
    keep = np.uint64(64) - rng.integers(12, 64, (2, n), dtype=np.uint64)
    man[:, : n // 4] = (man >> keep << keep)[:, : n // 4]
    man[:, n // 4: n // 2] |= ((np.uint64(1) << (np.uint64(52) - np.minimum(keep, 51))) -
                               np.uint64(1))[:, n // 4: n // 2]
    man &= np.uint64((1 << 52) - 1)
    ex = rng.integers(1023 - 480, 1023 + 480, (2, n), dtype=np.uint64)
    sg = rng.integers(0, 2, (2, n), dtype=np.uint64)
    x, y = ((sg << np.uint64(63)) | (ex << np.uint64(52)) | man).view(np.float64)
    tiny, big = 2.0 ** -1022, np.finfo(np.float64).max
    edge = np.array([0.0, -0.0, 1.0, -1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, tiny, -tiny,
                     big, 3.0, 1.0 / 3.0, 2.0 ** -64, 2.0 ** 64])
    a, b = (q.ravel() for q in np.meshgrid(edge, edge))
    with np.errstate(over="ignore", under="ignore"):
        p = np.abs(a * b)
    ok = (p == 0) & ((a == 0) | (b == 0)) | (p >= tiny) & np.isfinite(p)
    x, y = np.concatenate([x, a[ok]]), np.concatenate([y, b[ok]])
    got = nrd.check_softmul(dev(x), dev(y)).cpu().numpy()
    np.testing.assert_array_equal(got[0].view(np.uint64), got[1].view(np.uint64))
    np.testing.assert_array_equal(got[0].view(np.uint64), (x * y).view(np.uint64))
    # with the fallback: every operand, the ends of the range and nan included
    ends = np.array([5e-324, -3e-310, 1e-308, 1e308, -1e308, np.inf, -np.inf, np.nan, 0.0, 1.5])
    c, d = (q.ravel() for q in np.meshgrid(ends, ends))
    any_ = nrd.check_softmul(dev(np.concatenate([x, c])), dev(np.concatenate([y, d])))
    np.testing.assert_array_equal(any_[3].cpu().numpy(), any_[1].cpu().numpy())
    low = np.abs(x) < 2.0 ** 1000
    np.testing.assert_array_equal(got[2][low].view(np.uint64), (2 * x[low]).view(np.uint64))


HIERS = {
    "box16": lambda: W.uniform(16),
    "ragged": lambda: W.uniform((20, 12, 7)),
    "amr3": lambda: W.tiny_amr(8, True),
}


@pytest.mark.parametrize("outside", ["none", "some", "all"])
@pytest.mark.parametrize("tile", [(8, 8, 8), (32, 4, 4)])
@pytest.mark.parametrize("name", list(HIERS))
def test_window(nrd, name, tile, outside):
    h = HIERS[name]()
    z = W.material_from_cubes(h, [((2, 2, 2), 3, 10.0)])
    u = W.front_state(h, seed=2, noise=0.1)
    N = h.ncells
    rng = np.random.default_rng(4)
    if outside == "some":
        u[rng.integers(0, N, max(1, N // 40))] = 1e-22       # cold cells below 2^-64
    elif outside == "all":
        u[:N] *= 1e-21
    ctx = nrd.Context(nmg=1, tile_x=tile[0], tile_y=tile[1], tile_z=tile[2])
    ctx.set_hierarchy_from(h)
    ctx.set_material(dev(z))
    o = Oracle(h, z)
    b = u * (1 + 0.05 * rng.uniform(-1, 1, u.size))
    a0, dt = 1.5, 3e-3
    S = o.residual_scale(u, b, a0, dt)
    Fo = o.residual(u, b, a0, dt)
    F = ctx.residual(dev(u), dev(b), a0, dt)
    assert np.all(np.abs(F.cpu().numpy() - Fo) <= 1e-12 * S + 1e-300)
    # the linearisation's residual has the same bits
    assert torch.equal(ctx.linearise(dev(u), dev(b), a0, dt), F)
    v = W.random_direction(h, 7)
    J = ctx.jv(dev(u), dev(v), a0, dt, mode=nrd.JV_FROZEN).cpu().numpy()
    Sj = o.jv_scale(u, v, a0, dt)
    assert np.all(np.abs(J - o.jv_analytic(u, v, a0, dt)) <= 1e-12 * Sj + 1e-300)


VJP_HIERS = {
    "box8": lambda: W.uniform(8),
    "ragged": lambda: W.uniform((20, 12, 7)),
    "amr3": lambda: W.tiny_amr(8, True),
    "boundary": lambda: W.boundary_amr(8),     # patches on Robin and coarse-fine faces at once
}


@pytest.mark.parametrize("outside", ["none", "some", "all"])
@pytest.mark.parametrize("tile", [(8, 8, 8), (32, 4, 4)])
@pytest.mark.parametrize("name", list(VJP_HIERS))
def test_window_transpose(nrd, name, tile, outside):
    """The transposed product and the material partials with no, some and all
    cells outside the window, and both products on vectors whose entries leave
    the range of their integer products (2^-480 .. 2^480) and are zero."""
    h = VJP_HIERS[name]()
    z = W.material_from_cubes(h, [((2, 2, 2), 3, 10.0)])
    u = W.front_state(h, seed=2, noise=0.1)
    N = h.ncells
    rng = np.random.default_rng(4)
    if outside == "some":
        u[rng.integers(0, N, max(1, N // 40))] = 1e-22
    elif outside == "all":
        u[:N] *= 1e-21
    ctx = nrd.Context(nmg=1, tile_x=tile[0], tile_y=tile[1], tile_z=tile[2])
    ctx.set_hierarchy_from(h)
    ctx.set_material(dev(z))
    o = Oracle(h, z)
    a0, dt = 1.5, 3e-3
    ctx.linearise(dev(u), dev(u * 0.95), a0, dt)
    w = W.random_direction(h, 7)
    JTw, dz = ctx.vjp(dev(w), a0, dt)
    JTo, dzo, S = o.vjp(u, w, a0, dt)
    assert np.all(np.abs(JTw.cpu().numpy() - JTo) <= 1e-12 * S + 1e-300)
    assert np.abs(dz.cpu().numpy() - dzo).max() <= 1e-11 * np.abs(dzo).max()
    wide = w * 10.0 ** rng.choice([-200.0, -150.0, 0.0, 0.0, 160.0], w.size)
    wide[rng.integers(0, w.size, w.size // 10)] = 0.0
    JTw, _ = ctx.vjp(dev(wide), a0, dt, want_dz=False)
    JTo, _, S = o.vjp(u, wide, a0, dt, with_dz=False)
    assert np.all(np.abs(JTw.cpu().numpy() - JTo) <= 1e-12 * S + 1e-300)
    J = ctx.jv(dev(u), dev(wide), a0, dt, mode=nrd.JV_FROZEN).cpu().numpy()
    S = o.jv_scale(u, wide, a0, dt)
    assert np.all(np.abs(J - o.jv_analytic(u, wide, a0, dt)) <= 1e-12 * S + 1e-300)
