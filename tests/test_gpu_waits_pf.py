"""The P_F search's bounded waits, made to run out on purpose as test_gpu_waits.py does
for the U search: its loader issues no copies from one seed chunk on, so the MMA warp's
wait for that chunk, the epilogue's for its results and, in a short range, the loader's
own drain all end by their limit. The call reports bit 2, and the next one on the same
workspace gives the oracle's candidates."""
import numpy as np
import pytest
import torch

from gpu_util import assert_candidates_equal, oracle_encode, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,stall", [((4096, 512), 40), ((1000, 256), 6), ((1000, 256), 2), ((128, 64), 0)])
def test_bounded_wait_runs_out_and_is_reported(orc, shape, stall):
    import paper_2608_23144_gb300 as aw
    from synth import make_module
    m = make_module(*shape, seed=33, device="cpu", fisher=True, blend=(0.5, 0.5))
    kw = dict(C=64, P=4, b=4, S=4096, variant=1)
    prm, gm = aw.params(**kw), to_dev([m])
    before = aw.awsrc_encode_tiles(prm, gm)
    ws = before._awsrc_workspace
    assert aw.awsrc_workspace_status(ws) == 0
    before = before.clone()
    aw.awsrc_set_wait_test(200_000, stall)
    try:
        aw.awsrc_encode_tiles(prm, gm, workspace=ws)
        flags = aw.awsrc_workspace_status(ws)
    finally:
        aw.awsrc_set_wait_test()
    assert flags & 4, f"the timeout was not reported (flags {flags:#x})"
    after = aw.awsrc_encode_tiles(prm, gm, workspace=ws)
    assert aw.awsrc_workspace_status(ws) == 0
    assert torch.equal(after, before)
    n_cb = shape[1] // 64
    T = shape[0] * n_cb
    tiles = np.unique(np.concatenate([np.arange(min(T, 2 * n_cb)), np.arange(T - n_cb, T)]))
    want = oracle_encode(orc, orc.params(**kw), [m], tiles_per_module=[tiles])[0]
    assert_candidates_equal(aw.candidates_to_numpy(after)[tiles], want, f"after a timeout {shape}")
