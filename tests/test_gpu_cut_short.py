"""A step that a bounded device wait cut short concerns that step alone: its integrator
update is left out, the error is reported once by the next synchronising call, and the
frames enqueued meanwhile run as usual.  No wait expires here: the host writes the device
words that an expired wait would have written."""
import ctypes

import numpy as np
import pytest
import torch

import native

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")

POKE = """
#include "rtc_internal.h"
extern "C" int poke(rtc_handle* h, int word, int value) {
    return cudaMemcpy(h->d_status + word, &value, sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess ? 0 : 1;
}
extern "C" int timed_out() { return RTC_ETIMEDOUT; }
"""


@pytest.fixture(scope="module")
def poke(tmp_path_factory):
    import __graft_entry__ as g
    g.build()
    lib = native.compile_so(tmp_path_factory.mktemp("poke"), "poke", POKE)

    def f(r, word):
        torch.cuda.synchronize()
        assert lib.poke(r.handle, ctypes.c_int(word), ctypes.c_int(lib.timed_out())) == 0
    return f


def _pair(nsub, nact, store, pred):
    from paper_1805_07254_gb300.rtc import MLP_NPARAMS, Rtc
    rng = np.random.default_rng(nact)
    side, out = nsub * 4, []
    n = 2 * Rtc(nsub, 4, nact).info()["n_valid"]
    M = (rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
    p = (0.1 * rng.standard_normal(MLP_NPARAMS)).astype(np.float32)
    for _ in range(2):
        r = Rtc(nsub, 4, nact)
        r.load_calib(np.full((side, side), 5.0, np.float32), np.ones((side, side), np.float32))
        r.load_cmat(M, store=store)
        if pred:
            r.load_predictor(p, 0.3)
            r.set_predictor(True)
        out.append(r)
    frames = torch.from_numpy(rng.integers(0, 900, (5, side, side)).astype(np.uint16)).to(DEV)
    return out[0], out[1], frames


# 8x8: the last streaming block sums; 24x24: the sum kernel
@pytest.mark.parametrize("nsub,nact,store,pred", [(8, 69, "f32", False), (8, 69, "int8", True), (24, 460, "f32", False),
                                                  (24, 460, "bf16", True)])
def test_frames_after_an_expired_wait(poke, nsub, nact, store, pred):
    from paper_1805_07254_gb300.rtc import RtcError
    a, b, frames = _pair(nsub, nact, store, pred)
    st = torch.cuda.current_stream()
    dm = torch.zeros((5, nact), device=DEV)
    ref = torch.zeros((5, nact), device=DEV)
    for k in range(5):
        b.process_frame_async(frames[k], ref[k], stream=st)
    a.process_frame_async(frames[0], dm[0], stream=st)
    poke(a, 0)                                    # an earlier step's error, not yet taken
    for k in range(1, 5):
        a.process_frame_async(frames[k], dm[k], stream=st)
    with pytest.raises(RtcError):
        a.synchronize(st)                         # reported once
    a.synchronize(st)
    assert torch.equal(dm, ref)


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("nsub,nact,store", [(8, 69, "f32"), (24, 460, "f32"), (24, 460, "fp8")])
def test_only_the_marked_step_is_left_out(poke, nsub, nact, store, host):
    a, b, frames = _pair(nsub, nact, store, False)
    st = torch.cuda.current_stream()
    dm = torch.full((nact,), 7.0, device=DEV)
    ref = torch.zeros(nact, device=DEV)

    def step(k):
        if host:
            out = torch.full((nact,), 7.0).pin_memory()
            a.process_frame(frames[k].cpu().pin_memory(), dm_out=out)
            return out.to(DEV)
        dm.fill_(7.0)
        a.process_frame_async(frames[k], dm, stream=st)
        return dm.clone()

    step(0)
    b.process_frame_async(frames[0], ref, stream=st)
    before = a.get_dm()
    poke(a, 1)                                    # the mark of the step in flight
    assert torch.all(step(1) == 7.0)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a.get_dm(), before)
    for k in (2, 3):
        out = step(k)
        b.process_frame_async(frames[k], ref, stream=st)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    a.reconstruct_async(None, dm, stream=st)      # the stand-alone reconstruction too
    b.reconstruct_async(None, ref, stream=st)
    torch.cuda.synchronize()
    assert torch.equal(dm, ref)


def test_pageable_frame_reports_the_kept_state(poke):
    """A synchronous frame from pageable memory whose wait expired raises, its dm_out holds
    the state that was kept, and the next frame goes on from there."""
    from paper_1805_07254_gb300.rtc import RtcError
    a, b, frames = _pair(24, 460, "f32", False)
    f = frames.cpu().numpy()[:, None]
    first = a.process_frame(f[0])
    assert np.array_equal(first, b.process_frame(f[0]))
    poke(a, 0)
    poke(a, 1)
    out = np.full(460, 7.0, np.float32)
    with pytest.raises(RtcError):
        a.process_frame(f[1], dm_out=out)
    assert np.array_equal(out, first)
    assert np.array_equal(a.process_frame(f[2]), b.process_frame(f[2]))
