"""The decoder's three roundings fl(W0 + fl(fl(k_j C^-1/2) * scale)), where none of them
is exact: binary16 scales of full precision and C with an irrational C^-1/2, float32
weights in and out, so that a product fused into the sum would show."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["dense", "inplace"])
@pytest.mark.parametrize("C,P", [(8, 2), (8, 4), (32, 2), (32, 4), (128, 2), (128, 8), (256, 4), (64, 4)])
def test_three_roundings(orc, C, P, mode):
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(C + P)
    shapes = [(96, 512), (41, 256)]
    kw = dict(C=C, P=P, b=4, S=50, scale_mode=1, b_e=16)
    prm, oprm = aw.params(**kw), orc.params(**kw)
    W0 = [rng.normal(0, 0.02, s).astype(np.float32) for s in shapes]
    T = sum(w.size for w in W0) // C
    c = np.zeros(T, aw.CANDIDATE_DTYPE)
    c["gain"] = rng.random(T).astype(np.float32) + 0.1
    c["seed"] = rng.integers(0, 50, T)
    c["scale"] = rng.uniform(0.0005, 0.004, T).astype(np.float16).view(np.int16)
    c["code"][:, :P] = rng.integers(-7, 8, (T, P))
    stream, counts, _ = orc.select_records(oprm, shapes, c, [12.0])
    K = int(counts.sum())
    assert K == T
    want, bad = orc.decode_apply(oprm, W0, stream, K)
    assert bad == 0
    mods = [{"W0": torch.from_numpy(w).cuda()} for w in W0]
    st = torch.from_numpy(np.frombuffer(stream, np.uint8).copy()).cuda()
    if mode == "dense":
        outs = aw.awsrc_decode_apply(prm, mods, st, K, out_dtype=torch.float32)
    else:
        outs = [m["W0"].clone() for m in mods]
        aw.awsrc_decode_apply(prm, mods, st, K, outs=outs, out_dtype=torch.float32, mode=aw.DECODE_INPLACE)
    for o, w in zip(outs, want):
        assert np.array_equal(o.cpu().numpy(), w), np.abs(o.cpu().numpy() - w).max()
