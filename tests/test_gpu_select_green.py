"""Selection on a stream that may use few of the device's SMs (a green context): its
cooperative kernel takes no more blocks than those hold, and gives the same stream."""
import contextlib
import ctypes as ct

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _green_stream(sms):
    """A stream of a green context with about `sms` SMs of device 0 (driver API)."""
    cu = ct.CDLL("libcuda.so.1")

    def call(name, *args):
        if getattr(cu, name)(*args) != 0:
            pytest.skip(f"{name} is not available")
    resource = ct.c_uint64 * 18  # CUdevResource: type, padding, union at byte 96
    dev, whole, part, n = ct.c_int(), resource(), resource(), ct.c_uint(1)
    desc, ctx, st = ct.c_void_p(), ct.c_void_p(), ct.c_void_p()
    call("cuDeviceGet", ct.byref(dev), 0)
    call("cuDeviceGetDevResource", dev, ct.byref(whole), 1)
    call("cuDevSmResourceSplitByCount", ct.byref(part), ct.byref(n), ct.byref(whole), None, 0, sms)
    call("cuDevResourceGenerateDesc", ct.byref(desc), ct.byref(part), 1)
    call("cuGreenCtxCreate", ct.byref(ctx), desc, dev, 1)
    call("cuGreenCtxStreamCreate", ct.byref(st), ctx, 1, 0)
    assert ct.cast(part, ct.POINTER(ct.c_uint))[24] < 64  # SMs of the part
    yield torch.cuda.ExternalStream(st.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(st)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("variant", [0, 1])
def test_select_in_a_green_context(variant):
    import paper_2608_23144_gb300 as aw
    rng = np.random.default_rng(6)
    prm = aw.params(C=64, P=4, b=4, S=64, variant=variant)
    mods = [{"W0": torch.zeros(4096, 4096, dtype=torch.bfloat16, device="cuda")}] * 3
    c = np.zeros(3 * 4096 * 64, aw.CANDIDATE_DTYPE)
    c["gain"] = rng.random(len(c)).astype(np.float32)
    c["seed"] = rng.integers(0, 64, len(c))
    cands = torch.from_numpy(c.view(np.uint8).reshape(-1, 16).copy()).cuda()
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    want = [t.clone() for t in aw.awsrc_select_records(prm, mods, cands, [0.2], workspace=ws)]
    torch.cuda.synchronize()
    with _green_stream(16) as st:
        got = aw.awsrc_select_records(prm, mods, cands, [0.2], workspace=ws, stream=st)
        assert aw.awsrc_workspace_status(ws, st) == 0
    n = int(want[2][0])
    assert torch.equal(got[0][:n], want[0][:n]) and all(torch.equal(a, b) for a, b in zip(got[1:], want[1:]))
