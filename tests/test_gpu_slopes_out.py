"""Slopes written straight into the caller's buffer, and the buffers that still go
through a copy (a buffer not aligned to a float, one that overlaps the DM output): the
same bits in every case, from the stage call and from the frame call, and the resident
slope buffer is written as before."""
import numpy as np
import pytest
import torch

import synth
from helpers import make_pair

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


class _At:
    """A device address passed as a tensor-like object."""

    def __init__(self, ptr):
        self.ptr = ptr

    def data_ptr(self):
        return self.ptr

    def is_contiguous(self):
        return True


@pytest.mark.parametrize("npx,nsub,obs,n_wfs", [(8, 8, 0.0, 1), (7, 12, 0.2, 2), (10, 5, 0.0, 1), (16, 4, 0.0, 1)])
def test_direct_and_copied_slopes_agree(npx, nsub, obs, n_wfs):
    cfg = synth.tiny_scao().with_(name="s", nsub=nsub, npx=npx, obs=obs, dm_side=nsub + 1, n_wfs=n_wfs)
    frames, _ = synth.make_frames(cfg, 0, 3)
    r, oracle, *_ = make_pair(cfg)
    st = torch.cuda.current_stream()
    n, na = cfg.nslopes, cfg.nact
    raw = torch.zeros(4 * (n + na) + 64, dtype=torch.uint8, device=DEV)
    for k in range(3):
        f = frames[k].contiguous().to(DEV)
        _, s_ref = oracle.step(frames[k].numpy())
        s = torch.full((n + 2,), 9.0, device=DEV)
        r.centroid_async(f, s[1:n + 1], stream=st)               # direct, 4-byte aligned
        assert s[0] == 9.0 and s[n + 1] == 9.0
        assert np.max(np.abs(s[1:n + 1].cpu().numpy() - s_ref)) <= 1e-5
        r.centroid_async(f, _At(raw.data_ptr() + 1), stream=st)  # not float-aligned: copied
        got = raw[1:1 + 4 * n].cpu().numpy().tobytes()
        assert got == s[1:n + 1].cpu().numpy().tobytes()
        r.reset()
        dm, dm2 = torch.zeros(na, device=DEV), torch.zeros(na, device=DEV)
        r.reconstruct_async(None, dm, stream=st)                 # from the resident buffer
        r.synchronize(st)
        r.reset()
        s2 = torch.zeros(n, device=DEV)
        r.process_frame_async(f, dm2, s2, stream=st)
        assert torch.equal(s2, s[1:n + 1]) and torch.equal(dm, dm2)
        r.synchronize(st)
        r.reset()
        both = torch.zeros(n + na, device=DEV)                   # overlaps the DM output: copied last
        r.process_frame_async(f, both[:na], both[na // 2:na // 2 + n], stream=st)
        assert torch.equal(both[na // 2:na // 2 + n], s2)
        r.synchronize(st)
        r.reset()
        oracle.a[:] = 0
