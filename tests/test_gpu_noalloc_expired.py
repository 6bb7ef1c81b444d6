"""The allocation-free reconstruction when the copies of some blocks never land: their
rows keep the integrator state and their commands are NaN, the other rows are computed as
ever, and the next call goes on from the state that was kept.

The kernel is built here once more from its own source, with the copies of every third
block left out after their barrier was armed, so that nothing is in flight and the bounded
waits (200 ms each) run out."""
import ctypes

import numpy as np
import pytest
import torch

import native

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")

STALLED = """
#include "stream_mvm.cuh"
#define bulk_g2s(dst, src, bytes, bar, policy) if (blockIdx.x % 3 != 1) (bulk_g2s)(dst, src, bytes, bar, policy)
#include "mvm_noalloc.cu"
void rtc_set_global_error(const char*) {}
"""


@pytest.fixture(scope="module")
def stalled(tmp_path_factory):
    import __graft_entry__ as g
    g.build()
    f = native.compile_so(tmp_path_factory.mktemp("stalled"), "stalled", STALLED).rtc_mvm_integrate_noalloc
    f.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32, ctypes.c_void_p,
                  ctypes.c_void_p, ctypes.c_void_p, ctypes.c_float, ctypes.c_float, ctypes.c_int32, ctypes.c_void_p]
    return f


@pytest.mark.parametrize("with_dm", [True, False])
def test_rows_whose_copies_never_land(stalled, with_dm):
    from paper_1805_07254_gb300.rtc import DTYPES, mvm_integrate_noalloc
    nact, kpad = 600, 2064
    rng = np.random.default_rng(3)
    M = torch.from_numpy((rng.standard_normal((nact, kpad)) / kpad ** 0.5).astype(np.float32)).to(DEV)
    s = torch.from_numpy(rng.standard_normal(kpad).astype(np.float32)).to(DEV)
    a0 = torch.from_numpy(rng.standard_normal(nact).astype(np.float32)).to(DEV)
    want_a, want_dm = a0.clone(), torch.zeros(nact, device=DEV)
    mvm_integrate_noalloc(M, "f32", None, nact, kpad, s, want_a, want_dm)
    a, dm = a0.clone(), torch.full((nact,), 5.0, device=DEV)
    torch.cuda.synchronize()
    assert stalled(M.data_ptr(), DTYPES["f32"], None, nact, kpad, s.data_ptr(), a.data_ptr(),
                   dm.data_ptr() if with_dm else None, 0.4, 0.99, 1, None) == 0
    torch.cuda.synchronize()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = min(nact, sms)
    out = torch.zeros(nact, dtype=torch.bool, device=DEV)
    for b in range(1, blocks, 3):
        out[nact * b // blocks:nact * (b + 1) // blocks] = True
    assert torch.equal(a, torch.where(out, a0, want_a))
    if with_dm:
        assert torch.all(torch.isnan(dm[out])) and torch.equal(dm[~out], want_dm[~out])
    mvm_integrate_noalloc(M, "f32", None, nact, kpad, s, a, dm)
    torch.cuda.synchronize()
    assert torch.all(torch.isfinite(a)) and torch.equal(a, dm)
    again = want_a.clone()
    mvm_integrate_noalloc(M, "f32", None, nact, kpad, s, again, None)
    torch.cuda.synchronize()
    assert torch.equal(a, torch.where(out, want_a, again))
