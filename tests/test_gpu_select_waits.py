"""The selection's grid barriers, made to give up: with a limit of 1 ns a block that has
to wait at all leaves, and with it every other. The call reports bit 2 and returns, and
the next one on the same workspace gives the stream of an undisturbed call."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1])
def test_barrier_gives_up_and_is_reported(variant):
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(5)
    prm = aw.params(C=64, P=4, b=4, S=64, variant=variant)
    mods = [{"W0": torch.zeros(4096, 4096, dtype=torch.bfloat16, device="cuda")}] * 3
    c = np.zeros(3 * 4096 * 64, aw.CANDIDATE_DTYPE)
    c["gain"] = rng.random(len(c)).astype(np.float32)
    c["seed"] = rng.integers(0, 64, len(c))
    c["code"][:, :4] = rng.integers(-7, 8, (len(c), 4))
    cands = torch.from_numpy(c.view(np.uint8).reshape(-1, 16).copy()).cuda()
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")

    def select():
        out = aw.awsrc_select_records(prm, mods, cands, [0.2], workspace=ws)
        return [t.clone() for t in out]
    before = select()
    assert aw.awsrc_workspace_status(ws) == 0
    n = int(before[2][0])
    aw.awsrc_set_wait_test(1)
    try:
        select()
        flags = aw.awsrc_workspace_status(ws)
    finally:
        aw.awsrc_set_wait_test()
    assert flags & 4, f"the timeout was not reported (flags {flags:#x})"
    after = select()
    assert aw.awsrc_workspace_status(ws) == 0
    assert torch.equal(after[0][:n], before[0][:n]) and all(torch.equal(a, b) for a, b in zip(after[1:], before[1:]))
