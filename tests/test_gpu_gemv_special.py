"""The packed product of three to eight vectors on the tensor cores, against the
one-vector kernel and the oracle's double-precision definition: tile edges, and inputs
at the ends of binary32's range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _bound(cols, C, yabs):
    """The header's bound, without slack: (cols / min(C, 32) + 32) * 2^-24 * sum_j (|W0 x| + |r x|)."""
    return (cols / min(C, 32) + 32) * 2.0 ** -24 * yabs


def _setup(aw, orc, kw, W, recorded, scale, codes, rng, sdq=False):
    """Backbone of W, and a prepared sidecar that names the tiles of `recorded` (bool per tile)."""
    shapes = [W.shape]
    obb = orc.rtn_quantize(W, sdq=sdq)
    prm, oprm = aw.params(**kw), orc.params(**kw)
    T = W.size // prm.C
    c = np.zeros(T, aw.CANDIDATE_DTYPE)
    c["gain"][recorded] = 1.0
    c["seed"] = rng.integers(0, prm.S, T)
    c["scale"] = scale
    c["code"][:, :4] = codes(T)
    stream, counts, _ = orc.select_records(oprm, shapes, c, [40.0])
    K = int(counts.sum())
    assert K == recorded.sum()
    side = aw.awsrc_sidecar_prepare(prm, shapes, torch.from_numpy(np.frombuffer(stream, np.uint8).copy()).cuda(), K)
    bb = aw.awsrc_rtn_quantize(torch.from_numpy(W).cuda(), sdq=sdq)

    def gemv(x):
        return aw.awsrc_packed_gemv(prm, shapes, 0, bb, torch.from_numpy(x).cuda(), sidecar=side).cpu().numpy()

    def definition(x):
        y, yabs, bad = orc.packed_gemv(oprm, obb["q"], obb["s_eff"], 128, stream, K, x, shapes=shapes, m=0)
        assert bad == 0
        return y, yabs
    return gemv, definition


@pytest.mark.parametrize("kw,shape,M,sdq", [
    (dict(C=64, P=4, b=4, S=64), (1, 128), 3, True),
    (dict(C=64, P=4, b=4, S=64), (17, 256), 5, False),
    (dict(C=64, P=4, b=5, S=300), (33, 2432), 8, False),
    (dict(C=64, P=4, b=4, S=64), (130, 640), 3, True),
    (dict(C=32, P=4, b=4, S=32), (16, 1024), 6, True),
    (dict(C=32, P=4, b=4, S=32), (40, 384), 5, True),
    (dict(C=16, P=4, b=4, S=16), (31, 2176), 7, True),
    (dict(C=16, P=4, b=2, S=5), (129, 896), 4, False),
])
def test_tile_edges(orc, kw, shape, M, sdq):
    """Rows around a warp's 16, one to nineteen groups of columns (some of the eight sums
    empty, uneven ones) and every vector count."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(45 + M)
    W = rng.normal(0, 0.02, shape).astype(np.float32)
    q = 2 ** (kw["b"] - 1) - 1
    gemv, definition = _setup(aw, orc, kw, W, rng.random(W.size // kw["C"]) < 0.6, -8,
                              lambda T: rng.integers(-q, q + 1, (T, 4)), rng, sdq)
    x = rng.normal(0, 1, (M, shape[1])).astype(np.float32)
    x[0] *= 10.0 ** rng.uniform(-20, 20, shape[1]).astype(np.float32)  # every magnitude in one vector
    y = gemv(x)
    want, yabs = definition(x)
    assert (np.abs(y - want) <= _bound(shape[1], kw["C"], yabs)).all()


@pytest.mark.parametrize("C", [16, 32, 64])
def test_infinity_beside_recorded_tiles(orc, C):
    """Every other tile recorded, the infinities and NaN in tiles without a record: the
    recorded neighbour's row takes the backbone's infinity, or (scale 0) nothing."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(51)
    rows, cols, M = 48, 256, 5
    W = rng.normal(0, 0.02, (rows, cols)).astype(np.float32)
    W[::3, :128] = 0.0  # groups of scale 0
    even = np.arange(W.size // C) % 2 == 0
    gemv, _ = _setup(aw, orc, dict(C=C, P=4, b=4, S=64), W, even, -8, lambda T: rng.integers(-7, 8, (T, 4)), rng)
    x = rng.normal(0, 1, (M, cols)).astype(np.float32)
    clean = x.copy()
    x[1, C + 3] = np.inf
    x[2, 2 * C - 1] = -np.inf
    x[3, C] = np.nan
    y, yc = gemv(x), gemv(clean)
    one = np.concatenate([gemv(x[v:v + 1]) for v in range(M)])
    assert np.isfinite(one[1, ::3]).all() and np.isfinite(one[3, ::3]).all() and np.isinf(one[1]).any()
    for v in (0, 4):
        assert np.array_equal(y[v], yc[v])
    assert np.array_equal(np.isnan(y), np.isnan(one))
    assert np.array_equal(np.isposinf(y), np.isposinf(one)) and np.array_equal(np.isneginf(y), np.isneginf(one))
    fin = np.isfinite(one)
    assert np.allclose(y[fin], one[fin], rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("C,scale", [(64, -8), (64, 90), (32, -8), (16, 90)])
def test_small_inputs(orc, C, scale):
    """Inputs from 2^-100 down to the subnormals, where x has bits that BF16 does not:
    the header's bound relative to the products themselves (which large record scales
    bring back into the ordinary range). All of one sign, so that lost bits add up.
    Below the normal range each of the bound's roundings may also lose half of 2^-149."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(61)
    rows, cols, M = 40, 384, 8
    W = np.abs(rng.normal(0, 0.02, (rows, cols))).astype(np.float32) + np.float32(0.01)
    gemv, definition = _setup(aw, orc, dict(C=C, P=4, b=4, S=64), W, rng.random(W.size // C) < 0.5, scale,
                              lambda T: rng.integers(1, 8, (T, 4)), rng)
    x = rng.uniform(1, 2, (M, cols))
    x *= 2.0 ** np.array([-100, -108, -111, -114, -118, -122, -130, 0])[:, None]
    x[7] *= 2.0 ** rng.integers(-140, 1, cols)  # every magnitude in one vector
    x = x.astype(np.float32)
    y = gemv(x)
    want, yabs = definition(x)
    err = np.abs(y - want)
    assert (err <= _bound(cols, C, yabs) + (cols / min(C, 32) + 32) * 2.0 ** -150).all(), (err / yabs).max(1) * 2 ** 24


def test_large_inputs(orc):
    """Codes of 7 throughout and inputs at which a sum over a group's 128 codes and
    inputs would overflow, though one over 32 does not and the product, after the
    group's scale, is far from it."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(71)
    rows, cols, M, C = 40, 256, 3, 64
    W = np.full((rows, cols), 0.02, np.float32)
    gemv, definition = _setup(aw, orc, dict(C=C, P=4, b=4, S=64), W, rng.random(W.size // C) < 0.5, -10,
                              lambda T: rng.integers(-7, 8, (T, 4)), rng)
    x = rng.uniform(0.9e36, 1.2e36, (M, cols)).astype(np.float32)
    y = gemv(x)
    want, yabs = definition(x)
    assert np.isfinite(want).all() and np.isfinite(np.concatenate([gemv(x[v:v + 1]) for v in range(M)])).all()
    assert (np.abs(y - want) <= _bound(cols, C, yabs)).all()


@pytest.mark.parametrize("C", [16, 32, 64])
def test_largest_record_scale(orc, C):
    """The residual's operand k_j c 2^e near binary32's largest number (e = 126, and
    |k_j c| < 4) is finite, hence so is its product with small inputs."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(81)
    rows, cols, M = 40, 256, 3
    q = {16: 3, 32: 5, 64: 7}[C]  # |k_j| <= 4 q: k_j c up to 3, 3.5, 3.5
    W = rng.normal(0, 0.02, (rows, cols)).astype(np.float32)
    gemv, definition = _setup(aw, orc, dict(C=C, P=4, b=4, S=64), W, rng.random(W.size // C) < 0.5, 126,
                              lambda T: q * rng.choice([-1, 1], (T, 4)), rng)
    x = (rng.uniform(-1, 1, (M, cols)) * 2.0 ** -40).astype(np.float32)
    y = gemv(x)
    want, yabs = definition(x)
    assert np.isfinite(gemv(x[:1])).all() and np.abs(want).max() > 2.0 ** 80
    assert (np.abs(y - want) <= _bound(cols, C, yabs)).all()


@pytest.mark.parametrize("cols", [128, 384, 1152, 2048, 2432])
def test_bits_do_not_depend_on_the_batch(cols):
    """A product beside a task that fills the chip (fewer, longer column slices) has the
    bits of its single call (eight slices)."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(91)
    shapes, M = [(70000, 128), (50, cols)], 8
    prm = aw.params(C=64, P=4, b=4, S=64)
    bbs = [aw.awsrc_rtn_quantize(torch.from_numpy(rng.normal(0, 0.02, s).astype(np.float32)).cuda()) for s in shapes]
    xs = [torch.from_numpy(rng.normal(0, 1, (M, s[1])).astype(np.float32)).cuda() for s in shapes]
    both = aw.awsrc_packed_gemv_batch(prm, shapes, [(0, bbs[0], xs[0]), (1, bbs[1], xs[1])])
    for m in (0, 1):
        assert torch.equal(both[m], aw.awsrc_packed_gemv(prm, shapes, m, bbs[m], xs[m]))


@pytest.mark.parametrize("C", [16, 32, 64])
def test_smallest_record_scale(orc, C):
    """Records at e = -126 alone (a zero backbone): the operand k_j 2^(e - S) is a
    subnormal BF16, and the products with large inputs are in the ordinary range."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(85)
    rows, cols, M = 40, 256, 8
    W = np.zeros((rows, cols), np.float32)
    gemv, definition = _setup(aw, orc, dict(C=C, P=4, b=4, S=64), W, rng.random(W.size // C) < 0.5, -126,
                              lambda T: rng.integers(-7, 8, (T, 4)), rng)
    x = (rng.uniform(0.5, 1, (M, cols)) * 2.0 ** 110).astype(np.float32)
    y = gemv(x)
    want, yabs = definition(x)
    assert np.abs(want).max() > 2.0 ** -18
    assert (np.abs(y - want) <= _bound(cols, C, yabs)).all()
