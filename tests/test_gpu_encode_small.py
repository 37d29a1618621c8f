"""The mma.sync search (C in {16, 32, 64, 128}, P in {2, 4}) against the oracle,
every field bit for bit, where its tiling can go wrong: tile counts around a
warp's 16 and a block's 128, modules that end inside a warp's run, seed counts
around a group of eight and a shared-memory chunk, weight arrays off 16-byte
alignment, mixed dtypes, and tiles outside the numeric domain."""
import numpy as np
import pytest
import torch

from gpu_util import assert_candidates_equal, host_f32, oracle_encode

pytestmark = pytest.mark.gpu

U, PF = 0, 1
FP16 = dict(scale_mode=1, b_e=16)
NARROW = dict(b_e=4, e_bias=-9)  # exponents clamp: not the fast quantiser
CASES = [
    # params, (rows, cols) of the modules, dtypes (W, W0), elements off alignment
    (dict(C=16, P=4, S=16, variant=PF), [(7, 16), (1, 48), (130, 32), (3, 16)], ("bf16", "bf16"), 0),
    (dict(C=16, P=4, S=9, variant=PF), [(129, 16), (40, 48)], ("f32", "bf16"), 0),
    (dict(C=16, P=2, S=1, variant=PF), [(15, 16), (17, 32)], ("bf16", "bf16"), 3),
    (dict(C=16, P=4, S=200, variant=PF, **FP16), [(65, 32)], ("bf16", "f32"), 0),
    (dict(C=16, P=4, S=7, variant=U), [(16, 16), (113, 16), (1, 16)], ("f32", "f32"), 1),
    (dict(C=16, P=2, S=65, variant=U, **NARROW), [(33, 64)], ("bf16", "bf16"), 0),
    (dict(C=32, P=4, S=8, variant=PF, **NARROW), [(20, 64), (5, 32)], ("bf16", "bf16"), 0),
    (dict(C=32, P=2, S=130, variant=PF), [(64, 96)], ("bf16", "bf16"), 0),
    (dict(C=32, P=4, S=300, variant=U), [(70, 64)], ("f32", "f32"), 0),
    (dict(C=64, P=2, S=40, variant=U, **FP16), [(31, 128), (2, 64)], ("bf16", "bf16"), 5),
    (dict(C=64, P=2, S=24, variant=PF), [(50, 64)], ("f32", "bf16"), 0),
    (dict(C=128, P=2, S=2, variant=U), [(127, 128), (3, 256)], ("bf16", "bf16"), 0),
    (dict(C=128, P=4, S=33, variant=PF), [(30, 256)], ("bf16", "bf16"), 0),
    (dict(C=128, P=4, S=50, variant=U), [(40, 128)], ("f32", "f32"), 2),
    (dict(C=128, P=2, S=17, variant=PF, **FP16), [(18, 128)], ("bf16", "f32"), 0),
    (dict(C=16, P=4, S=16, variant=PF, ridge_rel=0.0, permute=0), [(60, 48)], ("bf16", "bf16"), 0),
]


def _off(t, n):
    """The tensor's values at an address n elements past an aligned one."""
    buf = torch.empty(t.numel() + n, dtype=t.dtype, device="cuda")
    out = buf[n:].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("case", range(len(CASES)))
def test_small_searches_match_oracle(orc, case):
    import paper_2608_23144_gb300 as aw
    from synth import make_module
    kw, shapes, (wd, w0d), off = CASES[case]
    kw = dict(dict(b=4), **kw)
    prm, oprm = aw.params(**kw), orc.params(**kw)
    dt = {"bf16": torch.bfloat16, "f32": torch.float32}
    mods = []
    for i, (r, c) in enumerate(shapes):
        m = make_module(r, c, seed=900 + 31 * case + i, device="cpu", w_dtype=wd, fisher=kw["variant"] == PF,
                        blend=(0.25, 0.75))
        m["W0"] = m["W0"].to(dt[w0d])
        C, T = prm.C, r * c // prm.C
        w = m["W"].view(T, C)
        w0 = m["W0"].view(T, C)
        if T > 12:  # degenerate tiles: no residual, one-hot, not finite, out of domain
            w[2].copy_(w0[2])
            w[5].copy_(w0[5])
            w[5, 3] += 0.5
            w[7, 1] = float("nan")
            w[9, 0] = 1e30
            w[11] = float("inf")
        mods.append(m)
    g = [{k: (_off(v, off) if torch.is_tensor(v) else v) for k, v in m.items()} for m in mods]
    got = aw.candidates_to_numpy(aw.awsrc_encode_tiles(prm, g))
    want = np.concatenate(oracle_encode(orc, oprm, mods))
    assert_candidates_equal(got, want, str(kw))


def test_small_search_many_tiles(orc):
    """More items than resident blocks, so that blocks reuse their tables (sampled rows)."""
    import paper_2608_23144_gb300 as aw
    from synth import make_module
    for kw in (dict(C=16, P=4, b=4, S=16, variant=PF), dict(C=128, P=2, b=4, S=2)):
        prm, oprm = aw.params(**kw), orc.params(**kw)
        m = make_module(3001, 2048, seed=5, device="cpu", fisher=prm.variant == PF, blend=(0.5, 0.5))
        g = {k: (v.cuda() if torch.is_tensor(v) else v) for k, v in m.items()}
        got = aw.candidates_to_numpy(aw.awsrc_encode_tiles(prm, [g]))
        n_cb = 2048 // prm.C
        tiles = np.concatenate([np.arange(n_cb), np.arange(1500 * n_cb, 1503 * n_cb), np.arange(3000 * n_cb, 3001 * n_cb)])
        want = orc.encode_tiles(oprm, host_f32(m["W"]), host_f32(m["W0"]), host_f32(m["act"]),
                                fisher=host_f32(m.get("fisher")), w_act=m["w_act"], w_fisher=m["w_fisher"], tiles=tiles)
        assert_candidates_equal(got[tiles], want, str(kw))
