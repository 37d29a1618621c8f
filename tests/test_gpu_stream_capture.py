"""The launch chains under stream capture (programmatic dependents in the encoder and
the decoder, the selection's cooperative launch, the product with several vectors): a
graph captured after one plain call of each gives the plain calls' bytes for inputs
that are replaced between the replays."""
import pytest
import torch

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(C=64, P=4, b=4, S=64),
    dict(C=64, P=4, b=4, S=64, variant=1),
    dict(C=16, P=4, b=4, S=16, variant=1),
    dict(C=128, P=2, b=4, S=2),
    dict(C=8, P=2, b=4, S=16),
])
def test_captured_chain_matches_plain_calls(kw):
    import paper_2608_23144_gb300 as aw
    from synth import make_module
    prm = aw.params(**kw)
    pf = prm.variant == 1
    draws = [to_dev([make_module(r, c, seed=s + i, device="cpu", fisher=pf, blend=(0.5, 0.5))
                     for i, (r, c) in enumerate([(150, 256), (33, 1024)])]) for s in (3, 40)]
    mods = [dict(m) for m in draws[0]]
    shapes = [tuple(m["W0"].shape) for m in mods]
    rates = [0.3, 0.6] if pf else [0.4]
    cap = aw.awsrc_stream_capacity(prm, mods, rates)
    T = sum(r * c // prm.C for r, c in shapes)
    new = dict(dtype=torch.uint8, device="cuda")
    cands, out = torch.empty((T, 16), **new), torch.empty(cap, **new)
    counts = torch.empty(len(rates) if pf else len(mods), dtype=torch.int64, device="cuda")
    nbytes = torch.empty(len(rates), dtype=torch.int64, device="cuda")
    ws = torch.empty(1 << 24, **new)
    W = [torch.empty_like(m["W0"]) for m in mods]
    bb = [aw.awsrc_rtn_quantize(m["W"], sdq=True) for m in mods]
    x = [torch.randn(5, c, device="cuda") for _, c in shapes]
    y = [torch.empty(5, r, device="cuda") for r, _ in shapes]

    def encode_select():
        out.zero_()  # only the stream's bytes are written
        aw.awsrc_encode_tiles(prm, mods, out=cands, workspace=ws)
        aw.awsrc_select_records(prm, mods, cands, rates, out=out, counts=counts, nbytes=nbytes, workspace=ws)

    def load(draw):
        for m, d in zip(mods, draw):
            for k in ("W", "W0", "act", "fisher"):
                if m.get(k) is not None:
                    m[k].copy_(d[k])

    mods = [{k: (v.clone() if torch.is_tensor(v) else v) for k, v in m.items()} for m in mods]
    K = None
    want = []
    for d in draws:
        load(d)
        encode_select()
        k = int(counts[0] if pf else counts.sum())
        K = k if K is None else min(K, k)
        want.append([t.clone() for t in (cands, out, counts, nbytes)])

    def apply():
        aw.awsrc_decode_apply(prm, mods, out, K, outs=W, workspace=ws)
        aw.awsrc_packed_gemv_batch(prm, shapes, [(i, bb[i], x[i], y[i]) for i in range(len(mods))])

    for d, w in zip(draws, want):
        load(d)
        encode_select()
        apply()
        w += [t.clone() for t in W + y]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(g, stream=side):
            encode_select()
            apply()
    torch.cuda.current_stream().wait_stream(side)
    for i in (0, 1, 0):
        load(draws[i])
        g.replay()
        torch.cuda.synchronize()
        for n, (a, b) in enumerate(zip([cands, out, counts, nbytes] + W + y, want[i])):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), (i, n)
    assert aw.awsrc_workspace_status(ws) == 0
