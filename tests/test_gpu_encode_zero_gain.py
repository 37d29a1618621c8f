"""P_F search where a tile's best gain is exactly zero: small whole-number residuals and
weights, codes of -1, 0 and 1 and one to four selectors, so that 2 sum q b and
sc q^T G q cancel to the last bit in some tiles. The gain is the recipe's +0."""
import numpy as np
import pytest
import torch

from gpu_util import assert_candidates_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,S", [(64, 1), (64, 2), (64, 4), (16, 1), (16, 2)])
def test_best_gain_zero(orc, C, S):
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(17 + S)
    rows, cols = 3000, 64
    r = ((rng.random((rows, cols)) < 0.03) * rng.integers(-1, 2, (rows, cols))).astype(np.float32)
    F = rng.integers(1, 3, (rows, cols)).astype(np.float32)
    W0, act = np.zeros_like(r), np.ones(cols, np.float32)
    kw = dict(C=C, P=4, b=2, S=S, variant=1)
    oprm = orc.params(**kw)
    want = orc.encode_tiles(oprm, r, W0, act, fisher=F, w_act=0.0, w_fisher=1.0, masks=orc.basis_masks(oprm))
    zero = (want["gain"] == 0) & np.any(want["code"] != 0, axis=1)
    assert zero.any() and (want["gain"][zero].view(np.uint32) == 0).all()
    m = {k: torch.from_numpy(v).cuda() for k, v in dict(W=r, W0=W0, act=act, fisher=F).items()}
    got = aw.awsrc_encode_tiles(aw.params(**kw), [dict(m, w_act=0.0, w_fisher=1.0)])
    assert aw.awsrc_workspace_status(got._awsrc_workspace) == 0
    assert_candidates_equal(aw.candidates_to_numpy(got), want, f"zero gains C={C} S={S}")
