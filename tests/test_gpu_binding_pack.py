"""The binding's one-pass argument packing gives the structs of the checked path,
byte for byte, and steps aside for anything that path would refuse or convert."""
import ctypes as ct

import pytest
import torch

pytestmark = pytest.mark.gpu


def _module(r, c, wd, w0d, fisher, act_extra=0):
    m = {"W": torch.randn(r, c, device="cuda").to(wd), "W0": torch.randn(r, c, device="cuda").to(w0d),
         "act": torch.rand(c + act_extra, device="cuda")}
    if fisher:
        m.update(fisher=torch.rand(r, c, device="cuda"), w_act=0.3, w_fisher=1e300)  # beyond binary32
    return m


def test_modules_pack_like_the_checked_path():
    from paper_2608_23144_gb300 import _binding as b
    bf, f32 = torch.bfloat16, torch.float32
    mods = [_module(3, 128, bf, bf, False), _module(5, 64, f32, bf, True), _module(1, 256, bf, f32, False, 7)]
    for dec in (False, True):
        arr, shapes = b._pack_modules(mods, dec)
        assert bytes(arr) == bytes(b.module_array(mods, dec))
        assert shapes == [(3, 128), (5, 64), (1, 256)]
    for bad in (dict(W=mods[0]["W"].float().t()), dict(act=mods[0]["act"].double()), dict(act=mods[0]["act"][:9]),
                dict(W0=mods[0]["W0"].cpu()), dict(W0=mods[0]["W0"].t()), dict(W=mods[0]["W"].half()),
                dict(fisher=torch.rand(3, 64, device="cuda"))):
        assert b._pack_modules([{**mods[0], **bad}], False) is None
    assert bytes(b._pack_shapes([(7, 128), (9, 64)])) == bytes(b.shape_modules([(7, 128), (9, 64)]))


@pytest.mark.parametrize("sdq", [False, True])
def test_gemv_and_backbone_tasks_pack_like_the_checked_path(sdq):
    from paper_2608_23144_gb300 import _binding as b
    shapes = [(40, 256), (24, 128)]
    Ws = [torch.randn(*s, device="cuda") for s in shapes]
    bbs = b.awsrc_rtn_quantize_batch(Ws, sdq=sdq)
    again = b._pack_rtn(Ws, sdq, bbs)
    want = (b.RtnTask * 2)()
    for i, (W, o) in enumerate(zip(Ws, bbs)):
        want[i] = b.RtnTask(W.shape[0], W.shape[1], W.data_ptr(), 0, int(sdq), o["codes"].data_ptr(),
                            o["scales"].data_ptr(), o["sdq_codes"].data_ptr() if sdq else None,
                            o["sdq_consts"].data_ptr() if sdq else None, o["W0"].data_ptr(), 0, 0)
    assert bytes(again) == bytes(want)
    xs = [torch.randn(3, c, device="cuda") for _, c in shapes]
    tasks = [(m, bbs[m], xs[m], torch.empty(3, shapes[m][0], device="cuda")) for m in (1, 0)]
    arr, ys, M, dev = b._pack_gemv(shapes, tasks)
    ref = (b.GemvTask * 2)()
    for i, (m, bb, x, y) in enumerate(tasks):
        ref[i] = b.GemvTask(m, 0, b._gemv_operands(shapes, m, bb, x, y)[2], x.data_ptr(), y.data_ptr())
    assert bytes(arr) == bytes(ref) and M == 3 and dev == 0 and ys == [t[3] for t in tasks]
    x = xs[0]
    for t in ((0, bbs[0], x.flatten()), (0, bbs[0], x.double()), (-1, bbs[0], x), (0, bbs[1], x), (0, bbs[0], x.t()),
              (0, bbs[0], x, torch.empty(3, 39, device="cuda")), (0, bbs[0], x[:, ::2])):
        assert b._pack_gemv(shapes, [t]) is None
    assert b._pack_gemv(shapes, [tasks[0], (0, bbs[0], x[:2])]) is None  # different numbers of vectors
    # the converted form still works: one vector given flat
    y0 = b.awsrc_packed_gemv(b.params(C=64, P=4, S=16), shapes, 0, bbs[0], x[0].clone())
    y1 = b.awsrc_packed_gemv(b.params(C=64, P=4, S=16), shapes, 0, bbs[0], x[:1].clone())
    assert torch.equal(y0, y1)
    assert ct.sizeof(b.Module) == 64
