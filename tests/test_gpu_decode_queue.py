"""The dense decoder's warp queues at the sizes where they can go wrong: modules whose
vectors end inside a lane, a warp's chunk of 128 and a block's 1024, no tile, every
tile and every other tile recorded, C from 8 to 256: the oracle's weights bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 256), (3, 256), (17, 512), (33, 256), (130, 768), (1, 2048), (2, 16384)]


@pytest.mark.parametrize("C,P,dtypes", [(64, 4, ("bf16", "bf16")), (8, 4, ("bf16", "f32")), (16, 2, ("f32", "bf16")),
                                        (256, 8, ("f32", "f32")), (32, 4, ("bf16", "bf16"))])
@pytest.mark.parametrize("pick", ["none", "all", "alternate", "first_and_last"])
def test_queue_edges_match_oracle(orc, C, P, dtypes, pick):
    import paper_2608_23144_gb300 as aw
    dt = {"bf16": torch.bfloat16, "f32": torch.float32}
    kw = dict(C=C, P=P, b=4, S=40)
    prm, oprm = aw.params(**kw), orc.params(**kw)
    rng = np.random.default_rng(C + P)
    T = sum(r * c // C for r, c in SHAPES)
    c = np.zeros(T, aw.CANDIDATE_DTYPE)
    sel = {"none": np.zeros(T, bool), "all": np.ones(T, bool), "alternate": np.arange(T) % 2 == 1,
           "first_and_last": (np.arange(T) == 0) | (np.arange(T) == T - 1)}[pick]
    c["gain"][sel] = rng.random(int(sel.sum())).astype(np.float32) + 0.1
    c["seed"] = rng.integers(0, 40, T)
    c["scale"] = rng.integers(-11, -6, T)
    c["code"][:, :P] = rng.integers(-7, 8, (T, P))
    stream, counts, _ = orc.select_records(oprm, SHAPES, c, [40.0])
    K = int(counts.sum())
    assert K == int(sel.sum())
    W0 = [torch.randn(r, k, generator=torch.Generator().manual_seed(r), dtype=torch.float32).to(dt[dtypes[0]]) * 0.02
          for r, k in SHAPES]
    mods = [{"W0": w.cuda()} for w in W0]
    outs = aw.awsrc_decode_apply(prm, mods, torch.from_numpy(np.frombuffer(stream, np.uint8).copy()).cuda(), K,
                                 out_dtype=dt[dtypes[1]])
    assert aw.awsrc_workspace_status(outs[0]._awsrc_workspace) == 0
    want, bad = orc.decode_apply(oprm, [w.float().numpy() for w in W0], stream, K, out_bf16=dtypes[1] == "bf16")
    assert bad == 0
    for o, w in zip(outs, want):
        assert np.array_equal(o.float().cpu().numpy(), w)
