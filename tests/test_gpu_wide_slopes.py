"""Slopes whose exact 16-bit parts would not hold all their bits: a huge slope where the
matrix is zero (a dead subaperture) beside ordinary ones, and slopes near the lower end
of FP32.  The commands are as near to the 64-bit product with the stored matrix as for
ordinary slopes: the tolerance is that of FP32 sums over the largest slice here (168
columns: 168 + 17 roundings of 2^-24 of the sum of magnitudes; the zero column adds
nothing to it), and the vector as a whole agrees to FP32 level.  The neighbouring slices
and the next call are unaffected, in the frame kernels and in the loop alike."""
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


def _handle(nact, n_wfs, store, seed, dead):
    from paper_1805_07254_gb300 import Rtc
    r = Rtc(20, 2, nact, n_wfs=n_wfs, gain=1.0, leak=1.0)
    n = r.info()["nslopes"]
    M = (np.random.default_rng(seed).standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
    M[:, [d % n for d in dead]] = 0.0
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
    assert np.all(np.abs(out - ref) <= (168 + 17) * 2.0 ** -24 * mag)
    assert np.linalg.norm(out - ref) <= 1e-6 * np.linalg.norm(mag)


@pytest.mark.parametrize("store", ["f32", "bf16", "f16", "fp8", "int8"])
@pytest.mark.parametrize("n_wfs,nact", [(1, 31), (6, 33), (9, 465), (20, 130), (40, 17)])
def test_a_huge_slope_where_the_matrix_is_zero(store, n_wfs, nact):
    dead = (5, -3)
    r, Ms, n = _handle(nact, n_wfs, store, n_wfs + nact, dead)
    s = (0.3 * np.random.default_rng(n_wfs).standard_normal(n)).astype(np.float32)
    clean = _reconstruct(r, s, nact)
    for v in (1e9, 1e13, 3e38):
        t = s.copy()
        t[list(dead)] = v, -v
        _check(_reconstruct(r, t, nact), Ms, t)
    assert np.array_equal(_reconstruct(r, s, nact), clean)


@pytest.mark.parametrize("store", ["f32", "bf16", "f16", "fp8", "int8"])
def test_tiny_slopes(store):
    r, Ms, n = _handle(65, 6, store, 3, ())
    rng = np.random.default_rng(4)
    for scale in (1e-24, 1e-31, 1e-35):
        s = (scale * (0.5 + rng.random(n))).astype(np.float32)
        _check(_reconstruct(r, s, 65), Ms, s)


@pytest.mark.parametrize("store", ["bf16", "f16", "int8"])
def test_the_loop_gives_the_same_bits(store):
    """Two pixels of one subaperture cancel in its flux but not in its moment: a slope of
    -3e15.  Frames and the persistent loop agree bit for bit, and with the 64-bit product
    of the measured slopes."""
    from paper_1805_07254_gb300 import Rtc
    nsub, npx, nact = 30, 4, 480
    side = nsub * npx
    rng = np.random.default_rng(6)
    flat = np.ones((1, side, side), np.float32)
    frames = rng.integers(1, 900, (3, 1, side, side)).astype(np.uint16)
    r = Rtc(nsub, npx, nact, gain=0.4, leak=0.99)
    y = np.arange(nsub) + 0.5 - nsub / 2
    sa = np.argwhere(y[:, None] ** 2 + y[None, :] ** 2 <= (nsub / 2) ** 2)
    n, i = r.info()["nslopes"], sa.shape[0] // 2
    assert n == 2 * sa.shape[0]
    row, col = sa[i] * npx
    frames[:, :, row:row + npx, col:col + npx] = 0
    frames[:, :, row, [col, col + 1, col + npx - 1]] = 1
    flat[0, row, col], flat[0, row, col + npx - 1] = 1e-15, -1e-15
    M = (rng.standard_normal((nact, n)) / np.sqrt(n)).astype(np.float32)
    M[:, [i, n // 2 + i]] = 0.0
    r.load_calib(np.zeros((1, side, side), np.float32), flat)
    r.load_cmat(M, store=store)
    r.set_threshold(0, -3e38)                      # nothing is clipped
    dm, s = r.process_frame(frames[0], want_slopes=True)
    assert s[i] < -1e15 and np.max(np.abs(np.delete(s, [i, n // 2 + i]))) < 10
    ref = 0.4 * (Q.stored_matrix(M, store).astype(np.float64) @ s.astype(np.float64))
    assert np.linalg.norm(dm - ref) <= 1e-6 * np.linalg.norm(ref)
    got = [dm] + [r.process_frame(frames[k]) for k in (1, 2)]
    r.reset()
    loop = []
    r.run_loop(3, frames=frames, sink=lambda k, d: loop.append(d))
    assert np.stack(loop).tobytes() == np.stack(got).tobytes()
