"""Where a job's DM commands go: a pinned buffer (written by the kernels), the middle of
one, and pageable memory (copied) receive the same bits, those of frames run alone; the
floats before and after are untouched.  Small systems whose last block sums, larger ones
with the sum kernel, the prediction, a handle without slopes."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("nsub,nact,store,pred", [(8, 69, "f32", False), (24, 460, "f32", False), (24, 460, "bf16", True),
                                                  (24, 460, "int8", False), (1, 5, "f32", False)])
def test_pinned_and_pageable_commands(nsub, nact, store, pred):
    from paper_1805_07254_gb300 import Rtc, Server
    from paper_1805_07254_gb300.rtc import MLP_NPARAMS, load_library
    lib, rng, side, n = load_library(), np.random.default_rng(nact), nsub * 4, 7
    r = Rtc(nsub, 4, nact, obs=0.9 if nsub == 1 else 0.0)
    m = r.info()["nslopes"]
    r.load_calib(np.full((side, side), 5.0, np.float32), np.ones((side, side), np.float32))
    r.load_cmat((rng.standard_normal((nact, m)) / np.sqrt(max(1, m))).astype(np.float32), store=store)
    if pred:
        r.load_predictor((0.1 * rng.standard_normal(MLP_NPARAMS)).astype(np.float32), 0.3)
        r.set_predictor(True)
    frames = torch.from_numpy(rng.integers(0, 900, (n, side, side)).astype(np.uint16))
    d, dm = frames.to(DEV), torch.zeros((n, nact), device=DEV)
    for k in range(n):
        r.process_frame_async(d[k].clone(), dm[k], stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    ref, pinned = dm.cpu().numpy(), frames.pin_memory()
    srv = Server(max_slots=3)
    for pin, off in ((True, 0), (True, 3), (False, 0)):
        r.reset()
        buf = torch.full((n * nact + 8,), 9.0)
        buf = buf.pin_memory() if pin else buf
        slot, done = ctypes.c_int32(-1), ctypes.c_uint64(0)
        assert lib.rtc_slot_submit(srv._h, r.handle, ctypes.c_void_p(pinned.data_ptr()), ctypes.c_uint64(n),
                                   ctypes.c_void_p(buf.data_ptr() + 4 * off), ctypes.byref(slot)) == 0
        while lib.rtc_slot_poll(srv._h, slot, ctypes.byref(done)) != 0:
            pass
        got = buf.numpy()
        assert got[off:off + n * nact].tobytes() == ref.tobytes()
        assert np.all(got[:off] == 9.0) and np.all(got[off + n * nact:] == 9.0)
    srv.close()
