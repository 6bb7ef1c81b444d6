"""Small systems, whose last streaming block sums the partial vectors, at the edges of its
groups of 32 rows and rounds of 128 and on both sides of the 16,384 partial values where
a kernel of its own takes over.  Frames from pinned host memory always use that kernel,
with the same order of additions, so both paths have to give the same bits, frame after
frame, enqueued one behind another and replayed from a graph."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _pair(nsub, npx, nact, store, pred):
    from paper_1805_07254_gb300.rtc import MLP_NPARAMS, Rtc
    rng = np.random.default_rng(nact)
    out = []
    for _ in range(2):
        r = Rtc(nsub, npx, nact)
        n = r.info()["nslopes"]
        if not out:
            M = (rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
            p = (0.1 * rng.standard_normal(MLP_NPARAMS)).astype(np.float32)
        side = nsub * npx
        r.load_calib(np.full((side, side), 5.0, np.float32), np.ones((side, side), np.float32))
        r.load_cmat(M, store=store)
        if pred:
            r.load_predictor(p, 0.3)
            r.set_predictor(True)
        out.append(r)
    return out


@pytest.mark.parametrize("pred", [False, True])
@pytest.mark.parametrize("nsub,npx,nact,store", [
    (2, 4, 1, "f32"), (8, 10, 31, "f32"), (8, 5, 32, "f16"), (8, 5, 33, "int8"), (8, 10, 69, "fp8"),
    (12, 5, 128, "bf16"), (12, 5, 129, "f32"), (10, 4, 204, "int8"), (14, 4, 107, "f32"), (14, 4, 108, "f32")])
def test_same_bits_as_the_sum_kernel(nsub, npx, nact, store, pred):
    a, b = _pair(nsub, npx, nact, store, pred)
    cfg = synth.tiny_scao().with_(name="s", nsub=nsub, npx=npx, obs=0.0, dm_side=nsub + 1)
    frames = synth.make_frames(cfg, 3, 6)[0]
    pinned, dm = frames.contiguous().pin_memory(), torch.zeros(nact).pin_memory()
    ref = np.stack([b.process_frame(pinned[k], dm_out=dm).numpy().copy() for k in range(6)])
    assert np.all(np.isfinite(ref)) and np.any(ref[5] != 0)
    d = frames.to(DEV)
    out = torch.zeros((6, nact), device=DEV)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    for k in range(3):
        a.process_frame_async(d[k], out[k], stream=st)
    if pred:                                    # the history ring's position is a launch argument
        for k in range(3, 6):
            a.process_frame_async(d[k], out[k], stream=st)
    else:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            for k in range(3, 6):
                a.process_frame_async(d[k], out[k], stream=torch.cuda.current_stream())
        g.replay()
    torch.cuda.synchronize()
    assert out.cpu().numpy().tobytes() == ref.tobytes()
