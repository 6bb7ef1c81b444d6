"""Matrix entries beyond the range of a 2-byte store are infinite there, and a command
that they enter is infinite with the sign of entry times slope, NaN where two of them
disagree or the slope is zero, as in FP32 arithmetic.  The other rows are unaffected.
Slices with a tail, of one 16-step and of several."""
import numpy as np
import pytest
import torch

from oracle import quant as Q

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("store,big", [("f16", 1e6), ("bf16", 3.4e38)])
@pytest.mark.parametrize("n_wfs", [1, 4, 9, 20])
def test_infinite_entries(store, big, n_wfs):
    from paper_1805_07254_gb300 import Rtc
    nact = 70
    r = Rtc(20, 2, nact, n_wfs=n_wfs, gain=1.0, leak=1.0)
    n = r.info()["nslopes"]
    rng = np.random.default_rng(n_wfs)
    M = (rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
    cols = sorted({0, 1, n // 3, n // 2 + 1, n - 1, *rng.integers(8, n, 20)})
    for i, c in enumerate(cols):                     # one infinite entry a row
        M[i, c] = big if i % 2 else -big
    k = len(cols)
    M[k, [5, 6]] = big, big                          # two that agree or not, by the slopes' signs
    M[k + 1, [5, n - 2]] = big, -big
    M[k + 2, 7] = big                                # meets a zero slope
    Ms = Q.stored_matrix(M, store).astype(np.float64)
    assert np.isinf(Ms).sum() == k + 5
    s = (0.3 * rng.standard_normal(n)).astype(np.float32)
    s[[3, 5]], s[6], s[7] = 0.5, -0.25, 0.0          # exact in one part; powers of two
    s[cols[2]] = 1.0
    r.load_cmat(M, store=store)
    out = torch.zeros(nact, device=DEV)
    r.reconstruct_async(torch.from_numpy(s).to(DEV), out, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    out = out.cpu().numpy().astype(np.float64)
    with np.errstate(invalid="ignore"):
        ref = Ms @ s.astype(np.float64)
    assert np.array_equal(np.isnan(out), np.isnan(ref)) and np.isnan(ref).sum() >= 1
    inf = np.isinf(ref)
    assert inf.sum() >= k and np.array_equal(out[inf], ref[inf])
    ok = np.isfinite(ref)
    mag = np.abs(Ms[ok]) @ np.abs(s.astype(np.float64))
    assert np.all(np.abs(out[ok] - ref[ok]) <= 4.1e-6 * mag)
