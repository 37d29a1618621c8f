"""Selection and serialisation at the sizes where the kernels' block split can go
wrong: record counts around a block's share, record widths from 3 to 16 bytes,
stream buffers at any byte offset, modules of one tile, few distinct gains, and
enough records for the largest block share. Bytes must equal the oracle's."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U, PF = 0, 1
SMALL = [(257, 16), (1, 16), (1023, 16), (640, 32)]   # C = 16: 2561 tiles, one module of one tile
CASES = [
    # kw, shapes, rates, byte offset of the stream buffer, distinct gains (0: all differ)
    (dict(C=16, P=1, b=2, S=1, b_e=1, variant=PF), SMALL, [1.2, 0.3], 0, 0),
    (dict(C=16, P=8, b=8, S=65536, scale_mode=1, b_e=16, variant=PF), SMALL, [3.2, 6.4, 6.41], 5, 0),
    (dict(C=16, P=4, b=4, S=16, variant=U), SMALL, [3.0], 3, 7),
    (dict(C=16, P=8, b=8, S=300, scale_mode=1, b_e=16, variant=U), SMALL, [8.0], 8, 0),
    (dict(C=16, P=4, b=4, S=4096, variant=PF), SMALL, [1.0, 2.0], 16, 1),
    (dict(C=4, P=2, b=3, S=9, variant=U), [(1, 4), (2048, 4), (2049, 8), (4095, 4)], [4.0], 1, 0),
    (dict(C=4, P=2, b=4, S=16, variant=PF), [(300001, 4), (1, 4), (512, 1024), (700000, 8)], [2.5, 8.0, 12.0], 7, 0),
    (dict(C=4, P=2, b=4, S=16, variant=U), [(300001, 4), (1, 4), (512, 1024), (700000, 8)], [9.0], 0, 3),
    # more tiles than a block compacts in one turn; four passes (every gain kept)
    (dict(C=4, P=4, b=4, S=4096, variant=PF), [(1 << 20, 16), (5001, 4), (64, 1024)], [1.3, 14.0], 5, 0),
    (dict(C=8, P=8, b=8, S=4096, scale_mode=1, b_e=16, variant=U), [(1 << 21, 8), ((1 << 21) + 77, 8)], [4.0], 0, 0),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_select_sizes_match_oracle(orc, case):
    import paper_2608_23144_gb300 as aw
    kw, shapes, rates, off, distinct = CASES[case]
    prm, oprm = aw.params(**kw), orc.params(**kw)
    T = sum(r * c // prm.C for r, c in shapes)
    rng = np.random.default_rng(17 + case)
    c = np.zeros(T, aw.CANDIDATE_DTYPE)
    gain = np.exp(rng.standard_normal(T) * 3.0).astype(np.float32)
    if distinct:
        gain = np.float32(0.5) + (rng.integers(0, distinct, T)).astype(np.float32)
    gain[rng.random(T) < 0.05] = -np.inf
    gain[rng.random(T) < 0.05] = 0.0
    gain[rng.random(T) < 0.02] = np.nan
    gain[rng.random(T) < 0.02] = np.float32(1e-42)    # subnormal gains are gains
    c["gain"] = gain
    c["seed"] = rng.integers(0, prm.S, T)
    c["scale"] = rng.integers(-2 ** (prm.b_e - 1), 2 ** (prm.b_e - 1), T)
    q = 2 ** (prm.b - 1) - 1
    c["code"][:, :prm.P] = rng.integers(-q, q + 1, (T, prm.P))
    mods = [{"W0": torch.empty(r, k, dtype=torch.bfloat16, device="cuda")} for r, k in shapes]
    dc = torch.from_numpy(c.view(np.uint8).reshape(-1, 16).copy()).cuda()
    cap = aw.awsrc_stream_capacity(prm, mods, rates)
    whole = torch.full((cap + off + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    stream, counts, nbytes = aw.awsrc_select_records(prm, mods, dc, rates, out=whole[off:off + cap])
    ostream, ocounts, obytes = orc.select_records(oprm, shapes, c, rates)
    assert list(counts.cpu().numpy()) == list(ocounts)
    assert list(nbytes.cpu().numpy()) == list(obytes)
    got = whole.cpu().numpy()
    n = int(max(obytes))
    assert bytes(got[off:off + n]) == ostream
    # nothing around the stream is written
    assert (got[:off] == 0xA5).all() and (got[off + n:] == 0xA5).all()
