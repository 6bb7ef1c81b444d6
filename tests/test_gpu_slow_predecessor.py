"""Frames enqueued behind a kernel that lets its successors start early and then runs for
longer than the bounded waits allow: the time counts for that kernel, not for the frame,
whose commands are those of a frame run alone."""
import ctypes

import numpy as np
import pytest
import torch

import native

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
BUSY_NS = 350_000_000          # the bounded waits of a frame are 200 ms

BUSY = """
#include "launch.cuh"
__global__ void busy_kernel(unsigned long long ns) {
    pdl_launch_dependents();
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int i = 0; i < 1000000; ++i) {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > ns) break;
    }
}
extern "C" int busy(void* st, unsigned long long ns) {
    busy_kernel<<<1, 32, 0, static_cast<cudaStream_t>(st)>>>(ns);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def busy(tmp_path_factory):
    import __graft_entry__ as g
    g.build()
    f = native.compile_so(tmp_path_factory.mktemp("busy"), "busy", BUSY).busy
    f.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong]
    return f


# prediction frames and frames of several pixel rounds a block request the whole ring
# early; the others one tile or none
@pytest.mark.parametrize("nsub,n_wfs,nact,store,pred", [(74, 1, 4421, "f32", True), (74, 1, 2000, "bf16", True),
                                                        (60, 4, 2900, "fp8", False), (74, 1, 4421, "f32", False),
                                                        (74, 1, 4421, "int8", False)])
def test_the_wait_for_the_predecessor_does_not_count(busy, nsub, n_wfs, nact, store, pred):
    from paper_1805_07254_gb300.rtc import MLP_NPARAMS, Rtc
    rng = np.random.default_rng(nact)
    side, pair = nsub * 4, []
    for _ in range(2):
        r = Rtc(nsub, 4, nact, n_wfs=n_wfs, obs=0.28)
        if not pair:
            n = r.info()["nslopes"]
            M = (rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
            p = (0.1 * rng.standard_normal(MLP_NPARAMS)).astype(np.float32)
        r.load_calib(np.full((n_wfs, side, side), 5.0, np.float32), np.ones((n_wfs, side, side), np.float32))
        r.load_cmat(M, store=store)
        if pred:
            r.load_predictor(p, 0.3)
            r.set_predictor(True)
        pair.append(r)
    frames = torch.from_numpy(rng.integers(0, 900, (2, n_wfs, side, side)).astype(np.uint16)).to(DEV)
    st = torch.cuda.Stream()
    dm, ref = torch.zeros((2, nact), device=DEV), torch.zeros((2, nact), device=DEV)
    torch.cuda.synchronize()
    for k in range(2):
        pair[1].process_frame_async(frames[k], ref[k], stream=st)
    pair[1].synchronize(st)
    pair[0].process_frame_async(frames[0], dm[0], stream=st)     # the plan and the code are there
    pair[0].synchronize(st)
    assert busy(st.cuda_stream, BUSY_NS) == 0
    pair[0].process_frame_async(frames[1], dm[1], stream=st)
    pair[0].synchronize(st)                                      # raises if a wait expired
    assert torch.equal(dm, ref)
