"""Selection over many modules of few tiles each, where the kernel has more blocks than
the tiles alone would give it (segments of one tile to several blocks' worth, more
segments than resident blocks, a large module among small ones): the oracle's stream."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("rows", [[1] * 3, [7] * 700, [1] * 1024, [5, 1, 9, 30] * 60, [3] * 40 + [9000] + [2] * 90])
def test_many_modules_match_oracle(orc, rows, variant):
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(len(rows))
    shapes = [(r, 64) for r in rows]
    kw = dict(C=64, P=4, b=4, S=100, variant=variant)
    prm, oprm = aw.params(**kw), orc.params(**kw)
    T = sum(rows)
    c = np.zeros(T, aw.CANDIDATE_DTYPE)
    c["gain"] = rng.integers(0, 50, T).astype(np.float32) / 7  # ties, and gains of zero
    c["seed"] = rng.integers(0, 100, T)
    c["scale"] = rng.integers(-11, -6, T)
    c["code"][:, :4] = rng.integers(-7, 8, (T, 4))
    want, counts, nbytes = orc.select_records(oprm, shapes, c, [12.0])
    mods = [{"W0": torch.zeros(s, dtype=torch.bfloat16, device="cuda")} for s in shapes]
    cands = torch.from_numpy(c.view(np.uint8).reshape(T, 16).copy()).cuda()
    out, k, b = aw.awsrc_select_records(prm, mods, cands, [12.0])
    assert list(k.cpu().numpy()) == list(counts) and list(b.cpu().numpy()) == list(nbytes)
    assert bytes(out.cpu().numpy()[: int(b[0])]) == want
