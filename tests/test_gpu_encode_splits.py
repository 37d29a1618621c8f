"""The mma.sync search on few tiles and many seeds, where its seed splits follow a rule
of their own: splits of one and of many groups of eight seeds, uneven last ones, one
block per SM and two; the oracle's candidates bit for bit."""
import numpy as np
import pytest

from gpu_util import assert_candidates_equal, oracle_encode, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,P,S,shape,variant", [
    (16, 2, 1024, (9, 64), 0), (16, 4, 777, (64, 64), 0), (16, 4, 2051, (16, 128), 1), (32, 2, 300, (130, 128), 1),
    (32, 4, 4096, (3, 64), 0), (64, 2, 1000, (20, 64), 0), (64, 2, 600, (40, 128), 1), (64, 2, 4000, (16, 64), 1),
    (128, 4, 1500, (10, 256), 1),
])
def test_candidates_match_oracle(orc, C, P, S, shape, variant):
    import paper_2608_23144_gb300 as aw
    from synth import make_module
    kw = dict(C=C, P=P, b=4, S=S, variant=variant)
    m = make_module(*shape, seed=C + P, device="cpu", fisher=bool(variant), blend=(0.5, 0.5))
    got = aw.awsrc_encode_tiles(aw.params(**kw), to_dev([m]))
    assert aw.awsrc_workspace_status(got._awsrc_workspace) == 0
    want = np.concatenate(oracle_encode(orc, orc.params(**kw), [m]))
    assert_candidates_equal(aw.candidates_to_numpy(got), want, f"{C} {P} {S} {shape} {variant}")
