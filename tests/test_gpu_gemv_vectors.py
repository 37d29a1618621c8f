"""The packed product on the tensor cores (three to eight vectors; C in {16, 32, 64},
P = 4, power-of-two scales) against the oracle's double-precision definition, within
the header's bound, where its tiling can go wrong: row counts around a warp's 16,
column slices of one to nineteen groups, every vector count, extreme scale exponents,
inputs over sixty decades, infinities and NaN."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _bound(cols, C, yabs):
    return (cols / min(C, 32) + 32) * 2.0 ** -24 * yabs + 1e-30


def _setup(aw, orc, kw, shapes, sdq, rng, rate=2.0, shift=0):
    """Backbones and an oracle stream over random candidates (exponents moved by `shift`)."""
    Ws = [rng.normal(0, 0.02, s).astype(np.float32) for s in shapes]
    obb = [orc.rtn_quantize(W, sdq=sdq) for W in Ws]
    prm, oprm = aw.params(**kw), orc.params(**kw)
    T = sum(r * c // prm.C for r, c in shapes)
    c = np.zeros(T, aw.CANDIDATE_DTYPE)
    c["gain"] = rng.random(T).astype(np.float32) + 0.1
    c["gain"][rng.random(T) < 0.3] = 0.0
    c["seed"] = rng.integers(0, prm.S, T)
    c["scale"] = rng.integers(-11, -6, T) + shift
    q = 2 ** (prm.b - 1) - 1
    c["code"][:, :4] = rng.integers(-q, q + 1, (T, 4))
    stream, counts, _ = orc.select_records(oprm, shapes, c, [rate])
    K = int(counts.sum())
    side = aw.awsrc_sidecar_prepare(prm, shapes, torch.from_numpy(np.frombuffer(stream, np.uint8).copy()).cuda(), K)
    bbs = [aw.awsrc_rtn_quantize(torch.from_numpy(W).cuda(), sdq=sdq) for W in Ws]
    return prm, oprm, obb, bbs, stream, K, side


@pytest.mark.parametrize("kw,shapes,M,sdq", [
    (dict(C=64, P=4, b=4, S=64), [(1, 128), (17, 256), (130, 640)], 3, True),
    (dict(C=64, P=4, b=5, S=300), [(33, 2432), (15, 1152)], 8, False),
    (dict(C=32, P=4, b=4, S=32), [(40, 384), (16, 1024)], 5, True),
    (dict(C=16, P=4, b=4, S=16), [(31, 2176), (129, 128)], 7, True),
    (dict(C=16, P=4, b=2, S=5), [(64, 896)], 4, False),
])
def test_vectors_match_definition(orc, kw, shapes, M, sdq):
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(21 + M)
    prm, oprm, obb, bbs, stream, K, side = _setup(aw, orc, kw, shapes, sdq, rng)
    for m, (rows, cols) in enumerate(shapes):
        x = rng.normal(0, 1, (M, cols)).astype(np.float32)
        x[0] *= 10.0 ** rng.uniform(-20, 20, cols).astype(np.float32)  # every magnitude in one vector
        for side_, K_ in ((side, K), (None, 0)):
            y = aw.awsrc_packed_gemv(prm, shapes, m, bbs[m], torch.from_numpy(x).cuda(), sidecar=side_).cpu().numpy()
            want, yabs, bad = orc.packed_gemv(oprm, obb[m]["q"], obb[m]["s_eff"], 128, stream, K_, x, shapes=shapes, m=m)
            assert bad == 0
            assert (np.abs(y - want) <= _bound(cols, kw["C"], yabs)).all(), (m, K_)


@pytest.mark.parametrize("C,shift", [(64, -113), (64, 100), (16, -113), (32, -110), (32, 90)])
def test_extreme_scales(orc, C, shift):
    """Exponents down to where 2^(e - 3) is a subnormal BF16, and large ones: the
    residual alone (a zero backbone) stays exact in its operands."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(31)
    shapes, M = [(48, 256)], 8
    kw = dict(C=C, P=4, b=4, S=64)
    prm, oprm, obb, bbs, stream, K, side = _setup(aw, orc, kw, shapes, False, rng, shift=shift)
    zero = dict(bbs[0], codes=torch.zeros_like(bbs[0]["codes"]))
    x = (rng.normal(0, 1, (M, 256)) * 2.0 ** -shift).astype(np.float32)
    y = aw.awsrc_packed_gemv(prm, shapes, 0, zero, torch.from_numpy(x).cuda(), sidecar=side).cpu().numpy()
    want, yabs, bad = orc.packed_gemv(oprm, np.zeros_like(obb[0]["q"]), obb[0]["s_eff"], 128, stream, K, x,
                                      shapes=shapes, m=0)
    assert bad == 0 and np.abs(want).max() > 1e-6
    assert (np.abs(y - want) <= _bound(256, C, yabs)).all()


def test_infinities_and_nan(orc):
    """Vectors with a non-finite or huge input: every y has the class (finite,
    infinity of a sign, NaN) that the one-vector kernel gives on the FP32 pipes;
    the other vectors are unaffected."""
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(41)
    shapes, M = [(64, 512)], 6
    prm, oprm, obb, bbs, stream, K, side = _setup(aw, orc, dict(C=64, P=4, b=4, S=64), shapes, True, rng, rate=0.5)
    x = rng.normal(0, 1, (M, 512)).astype(np.float32)
    clean = x.copy()
    x[1, 100] = np.inf
    x[2, 7] = -np.inf
    x[3, 300] = np.nan
    x[4, 511] = np.float32(3.4e38)

    def gemv(v):
        return aw.awsrc_packed_gemv(prm, shapes, 0, bbs[0], torch.from_numpy(v).cuda(), sidecar=side).cpu().numpy()
    y, yc = gemv(x), gemv(clean)
    one = np.concatenate([gemv(x[v:v + 1]) for v in range(M)])
    for v in (0, 5):
        assert np.array_equal(y[v], yc[v])
    assert np.array_equal(np.isnan(y), np.isnan(one))
    assert np.array_equal(np.isposinf(y), np.isposinf(one)) and np.array_equal(np.isneginf(y), np.isneginf(one))
    assert np.isinf(y[1]).any() and np.isnan(y[1]).any() and np.isnan(y[3]).all()
    fin = np.isfinite(one[4])
    assert np.allclose(y[4][fin], one[4][fin], rtol=1e-5, atol=np.abs(one[4][fin]).max() * 1e-6)
