"""A server of 32 slots gives each job 4 of the SMs: a block then has some 40 slices, and
the padding of each slice's slopes to 16 must not refuse a system that fits without it
(72x72 subapertures of four sensors, 8,144 slopes a block).  Same bits as on all SMs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("store", ["f32", "bf16", "f16", "fp8", "int8"])
def test_many_slices_a_block(store):
    from paper_1805_07254_gb300 import Rtc, Server
    nact, side = 23, 144
    rng = np.random.default_rng(5)
    r = Rtc(72, 2, nact, n_wfs=4)
    n = r.info()["nslopes"]
    r.load_calib(np.full((4, side, side), 5.0, np.float32), np.ones((4, side, side), np.float32))
    r.load_cmat((rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32), store=store)
    frames = rng.integers(0, 900, (3, 4, side, side)).astype(np.uint16)
    d, dm = torch.from_numpy(frames).to(DEV), torch.zeros((3, nact), device=DEV)
    for k in range(3):
        r.process_frame_async(d[k], dm[k], stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    r.reset()
    srv = Server(max_slots=32)
    got = srv.wait(srv.submit(r, frames))
    srv.close()
    assert np.asarray(got).tobytes() == dm.cpu().numpy().tobytes() and np.any(got != 0)
