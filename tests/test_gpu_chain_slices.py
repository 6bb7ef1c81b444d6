"""Small slices of 1- and 2-byte stores, which go by FP32 chains, on both sides of the line
to the tensor cores (40 columns times rows a thread, 90 for INT8): every tail (2 to 44 columns), one
row and rows around a thread's second and third, one and several slices a block (a
server's share of the SMs), the prediction.  The tolerance is that of FP32 sums: 44 + 17
roundings of 2^-24 of the sum of magnitudes.  Infinite, NaN and huge slopes, frames, the
stand-alone reconstruction, the loop and a server slot all agree bit for bit."""
import numpy as np
import pytest
import torch

import synth
from oracle import quant as Q

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
STORES = ["bf16", "f16", "fp8", "int8"]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _reconstruct(r, s, nact):
    out = torch.zeros(nact, device=DEV)
    r.reset()
    r.reconstruct_async(torch.from_numpy(s).to(DEV), out, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    return out.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("store", STORES)
@pytest.mark.parametrize("nsub,n_wfs,nact", [(2, 1, 1), (16, 1, 17), (20, 2, 448), (20, 3, 449), (20, 4, 897),
                                             (20, 5, 1344), (20, 9, 33), (20, 9, 448), (20, 9, 449), (20, 10, 31),
                                             (20, 10, 896), (20, 8, 1344)])
def test_reconstruction(store, nsub, n_wfs, nact):
    from paper_1805_07254_gb300 import Rtc
    r = Rtc(nsub, 2, nact, n_wfs=n_wfs, gain=1.0, leak=1.0)
    n = r.info()["nslopes"]
    rng = np.random.default_rng(10 * n_wfs + nact)
    M = (rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
    r.load_cmat(M, store=store)
    Ms = Q.stored_matrix(M, store).astype(np.float64)
    s = (0.3 * rng.standard_normal(n)).astype(np.float32)
    out = _reconstruct(r, s, nact)
    mag = np.abs(Ms) @ np.abs(s.astype(np.float64))
    assert np.all(np.abs(out - Ms @ s.astype(np.float64)) <= (44 + 17) * 2.0 ** -24 * mag)
    for v in (np.inf, -np.inf, np.nan):
        t = s.copy()
        t[n // 2] = v
        with np.errstate(invalid="ignore"):
            ref = Ms @ t.astype(np.float64)
        got = _reconstruct(r, t, nact)
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
    assert np.array_equal(_reconstruct(r, s, nact), out)


@pytest.mark.parametrize("pred", [False, True])
@pytest.mark.parametrize("store", STORES)
@pytest.mark.parametrize("nsub,npx,nact", [(8, 10, 69), (26, 4, 560), (34, 4, 940)])
def test_frames_loop_and_slot_agree(nsub, npx, nact, store, pred):
    from paper_1805_07254_gb300 import Rtc, Server
    from paper_1805_07254_gb300.rtc import MLP_NPARAMS
    rng = np.random.default_rng(nact)
    cfg = synth.tiny_scao().with_(name="s", nsub=nsub, npx=npx, obs=0.0, dm_side=nsub + 1)
    frames = synth.make_frames(cfg, 3, 5)[0]
    side = nsub * npx
    r = Rtc(nsub, npx, nact)
    n = r.info()["nslopes"]
    r.load_calib(np.full((side, side), 5.0, np.float32), np.ones((side, side), np.float32))
    r.load_cmat((rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32), store=store)
    if pred:
        r.load_predictor((0.1 * rng.standard_normal(MLP_NPARAMS)).astype(np.float32), 0.3)
        r.set_predictor(True)
    st = torch.cuda.current_stream()
    d, dm = frames.to(DEV), torch.zeros((5, nact), device=DEV)
    for k in range(5):
        r.process_frame_async(d[k], dm[k], stream=st)
    torch.cuda.synchronize()
    ref = dm.cpu().numpy()
    assert np.all(np.isfinite(ref)) and np.any(ref[4] != 0)
    pinned, out = frames.contiguous().pin_memory(), torch.zeros(nact).pin_memory()
    r.reset()
    host = np.stack([r.process_frame(pinned[k], dm_out=out).numpy().copy() for k in range(5)])
    r.reset()
    loop = []
    r.run_loop(5, frames=frames.numpy(), sink=lambda k, a: loop.append(a))
    r.reset()
    srv = Server(max_slots=16)
    slot = srv.wait(srv.submit(r, frames.numpy()))
    srv.close()
    for got in (host, np.stack(loop), slot):
        assert np.asarray(got).tobytes() == ref.tobytes()
