"""The tcgen05 P_F search works on the integer sums themselves while a block's grids,
its pivots and its fits stay inside fixed ranges, and in the recipe's units otherwise.
Weights and residuals scaled across those ranges (all rows, or some rows of a block),
rows without residual or weight, and near-singular tiles: the oracle's candidates bit
for bit either way."""
import numpy as np
import pytest
import torch

from gpu_util import assert_candidates_equal, oracle_encode, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wexp,rexp,some_rows", [
    (0, 0, False), (-9, 0, False), (-11, 0, False), (-40, 0, False), (30, 0, False), (36, -3, False),
    (0, -18, False), (0, -24, False), (0, -60, False), (-30, 8, True), (-12, -20, True), (25, -30, True),
])
def test_scaled_tiles_match_oracle(orc, wexp, rexp, some_rows):
    import paper_2608_23144_gb300 as aw
    from synth import make_module
    kw = dict(C=64, P=4, b=4, S=100, variant=1)
    prm, oprm = aw.params(**kw), orc.params(**kw)
    m = make_module(150, 128, seed=77, device="cpu", w_dtype="f32", fisher=True, blend=(0.5, 0.5))
    rows = torch.arange(150) % 7 == 3 if some_rows else torch.ones(150, dtype=torch.bool)
    m["w_act"] = 0.0 if some_rows else float(np.float32(m["w_act"] * 2.0 ** wexp))
    m["fisher"][rows] *= 2.0 ** wexp
    m["W"] = m["W"].clone()
    m["W"][rows] = m["W0"][rows] + (m["W"] - m["W0"])[rows] * 2.0 ** rexp
    m["W"][11] = m["W0"][11]                      # no residual
    m["fisher"][13] = 0.0                         # weights of the activations alone, or none
    m["fisher"][17] *= (torch.rand(128) < 0.05)   # few weights: nearly singular Gram matrices
    m["fisher"][19, 5] *= 2.0 ** 30               # one weight above all others
    m["W"][23, 70] = float("inf")
    got = aw.candidates_to_numpy(aw.awsrc_encode_tiles(prm, to_dev([m])))
    want = np.concatenate(oracle_encode(orc, oprm, [m]))
    assert_candidates_equal(got, want, f"{wexp} {rexp} {some_rows}")
