"""Reconstruction from 1- and 2-byte stores on the tensor cores, at the edges of its
layout: slices of 2 to 168 columns (tails of every length, one 16-step, several 32s),
row counts around the groups of 16 and the tiles of 448, FP32 beside them.

Products of a stored value and a slope's part are exact, so a command differs from the
64-bit product with the stored matrix by FP32 accumulation alone: at most K / 16 + 2
accumulation steps of 2^-22 of the partial sum's magnitude per slice, and 11 + 4 + 2
FP32 additions of 2^-24 over the slices and the integrator.  For the widest slices here
(K = 168) that is 13 x 2.4e-7 + 17 x 6e-8 = 4.1e-6 of the largest partial; the tolerance is
4.1e-6 of the vector's RMS times the cancellation between slices, which the sum of
magnitudes bounds."""
import numpy as np
import pytest
import torch

from oracle import quant as Q

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
STORES = ["f32", "bf16", "f16", "fp8", "int8"]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _handle(nact, n_wfs, store, seed, nsub=20):
    from paper_1805_07254_gb300 import Rtc
    r = Rtc(nsub, 2, nact, n_wfs=n_wfs, gain=1.0, leak=1.0)
    n = r.info()["nslopes"]
    M = (np.random.default_rng(seed).standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
    r.load_cmat(M, store=store)
    return r, Q.stored_matrix(M, store).astype(np.float64), n


def _reconstruct(r, s, nact):
    out = torch.zeros(nact, device=DEV)
    r.reset()
    r.reconstruct_async(torch.from_numpy(s).to(DEV), out, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    return out.cpu().numpy().astype(np.float64)


def _check(out, Ms, s):
    ref = Ms @ s.astype(np.float64)
    mag = np.abs(Ms) @ np.abs(s.astype(np.float64))
    assert np.all(np.abs(out - ref) <= 4.1e-6 * mag + 1e-37), np.max(np.abs(out - ref) / mag)
    # and far nearer than that on the whole: FP32-level agreement of the vector
    assert np.linalg.norm(out - ref) <= 1e-6 * np.linalg.norm(mag)


@pytest.mark.parametrize("store", STORES)
@pytest.mark.parametrize("n_wfs,nact", [(1, 1), (1, 449), (2, 15), (3, 16), (4, 17), (5, 31), (6, 33), (8, 448),
                                        (11, 900), (13, 47), (15, 64), (40, 130)])
def test_reconstruction_matches_the_stored_matrix(store, n_wfs, nact):
    r, Ms, n = _handle(nact, n_wfs, store, 100 * n_wfs + nact)
    s = (0.3 * np.random.default_rng(n_wfs).standard_normal(n)).astype(np.float32)
    out = _reconstruct(r, s, nact)
    _check(out, Ms, s)
    assert np.array_equal(out, _reconstruct(r, s, nact))


@pytest.mark.parametrize("store", STORES)
def test_slopes_of_any_magnitude(store):
    """Slopes 24 orders of magnitude apart, within a slice and between slices."""
    r, Ms, n = _handle(65, 6, store, 7)
    rng = np.random.default_rng(8)
    for lo, hi in ((-12, 12), (-30, -25), (25, 30), (-36, -34)):
        s = (rng.standard_normal(n) * 10.0 ** rng.uniform(lo, hi, n)).astype(np.float32)
        _check(_reconstruct(r, s, 65), Ms, s)
    s = np.zeros(n, np.float32)
    assert np.all(_reconstruct(r, s, 65) == 0)


@pytest.mark.parametrize("store", STORES)
def test_infinite_and_nan_slopes(store):
    """One infinite slope makes the commands infinite (NaN where the matrix is zero
    there), a NaN one makes them NaN, as in FP32 arithmetic; the next call is clean."""
    r, Ms, n = _handle(65, 6, store, 9)
    s = (0.3 * np.random.default_rng(10).standard_normal(n)).astype(np.float32)
    clean = _reconstruct(r, s, 65)
    for at in (0, n // 2 + 3, n - 1):
        for v in (np.inf, -np.inf, np.nan):
            t = s.copy()
            t[at] = v
            with np.errstate(invalid="ignore"):
                ref = Ms @ t.astype(np.float64)
            out = _reconstruct(r, t, 65)
            assert np.array_equal(np.isnan(out), np.isnan(ref))
            assert np.array_equal(out[np.isinf(ref)], ref[np.isinf(ref)])
    assert np.array_equal(_reconstruct(r, s, 65), clean)
