"""Frames of several handles one behind another on one stream, where each launch may start
while the one before it drains: a streaming kernel of one handle behind the sum of
another, a pixel kernel behind either, the allocation-free reconstruction and the
predictor's training among them.  The same bits as each handle by itself."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _handle(nsub, nact, store, pred, seed):
    from paper_1805_07254_gb300.rtc import MLP_NPARAMS, Rtc
    rng = np.random.default_rng(seed)
    r, side = Rtc(nsub, 4, nact), nsub * 4
    n = r.info()["nslopes"]
    r.load_calib(np.full((side, side), 5.0, np.float32), np.ones((side, side), np.float32))
    r.load_cmat((rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32), store=store)
    if pred:
        r.load_predictor((0.1 * rng.standard_normal(MLP_NPARAMS)).astype(np.float32), 0.3)
        r.set_predictor(True)
    frames = torch.from_numpy(rng.integers(0, 900, (12, side, side)).astype(np.uint16)).to(DEV)
    return r, frames, torch.zeros((12, nact), device=DEV), torch.zeros((12, n), device=DEV)


def test_handles_interleaved_on_one_stream():
    from paper_1805_07254_gb300 import Mlp
    from paper_1805_07254_gb300.rtc import mvm_integrate_noalloc
    from synth.mlp_init import flatten, init_mlp_params
    hs = [_handle(*a) for a in ((8, 69, "f32", False, 1), (40, 1300, "f32", False, 2), (24, 460, "int8", True, 3),
                                (40, 1300, "bf16", False, 4), (10, 80, "f16", True, 5), (56, 2500, "fp8", False, 6))]
    M = torch.randn((900, 1104), device=DEV) / 33.0
    s = torch.randn(1104, device=DEV)
    X, T = torch.randn((300, 200), device=DEV), torch.randn((300, 2), device=DEV)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    results = []
    for mixed in (False, True):
        net = Mlp(params=flatten(init_mlp_params(3)))
        a, dm = torch.zeros(900, device=DEV), torch.zeros((12, 900), device=DEV)
        for r, _, out, sl in hs:
            r.reset()
            out.zero_()
            sl.zero_()
        torch.cuda.synchronize()

        def frame(h, k):
            r, f, out, sl = h
            r.process_frame_async(f[k], out[k], sl[k] if k % 2 else None, stream=st)

        def rest(k):
            mvm_integrate_noalloc(M, "f32", None, 900, 1104, s, a, dm[k], stream=st)
            net.train_step(X, T, 1e-3, stream=st)
        if mixed:
            for k in range(12):
                for h in hs:
                    frame(h, k)
                    if k % 3 == 0:
                        h[0].centroid_async(h[1][k], h[3][k], stream=st)
                rest(k)
        else:
            for h in hs:
                for k in range(12):
                    frame(h, k)
                    torch.cuda.synchronize()
                    if k % 3 == 0:
                        h[0].centroid_async(h[1][k], h[3][k], stream=st)
                    torch.cuda.synchronize()
            for k in range(12):
                rest(k)
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        results.append([t.cpu().clone() for h in hs for t in h[2:]] + [a.cpu(), dm.cpu(), torch.from_numpy(net.get_params())])
    for x, y in zip(*results):
        assert torch.equal(x, y)
    assert all(torch.any(x != 0) for x in results[0])
