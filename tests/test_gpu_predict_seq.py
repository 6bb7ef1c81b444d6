"""The sequence predictor kernel at the edges of its split: tiles of 32 subapertures
(one, a remainder, a whole tile, one more), runs of frames shorter and longer than a
warp's share, and an output that overlaps the sequence.

Every row of a long call must equal, bit for bit, the row that a 5-frame call (one
predicted frame) gives: no ring slot, tile or run boundary may show.  The 5-frame rows
are held to the oracle at the device's rounding points with the tolerance of
tests/test_gpu_mlp.py: 1e-5 of the largest |y| (FP32 arithmetic), the effect of every h1
entry that may round the other way, and the ulp of the result."""
import numpy as np
import pytest
import torch

import mlp_emul as E
from oracle import mlp as L
from synth.mlp_init import flatten, init_mlp_params

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _net(nv, nsub, seed):
    from paper_1805_07254_gb300 import Mlp
    rng = np.random.default_rng(seed)
    cells = np.sort(rng.choice(nsub * nsub, nv, replace=False))
    rc = np.stack([cells // nsub, cells % nsub], axis=1).astype(np.int32)
    params = init_mlp_params(seed)
    m = Mlp(params=flatten(params))
    m.set_geometry(rc, nsub)
    return m, rc, params, rng


def _one(m, S, k, sigma):
    """Row k + 1 of the prediction from the five rows k-3 .. k+1 alone."""
    out = torch.zeros((5, S.shape[1]), device=DEV)
    m.predict_seq(S[k - 3:k + 2].contiguous(), sigma, out)
    return out[4]


@pytest.mark.parametrize("nv,nsub,n", [(1, 4, 5), (31, 8, 40), (32, 8, 6), (33, 8, 41), (52, 8, 2500), (700, 30, 90)])
def test_rows_do_not_depend_on_the_split(nv, nsub, n):
    m, rc, params, rng = _net(nv, nsub, 40 + nv)
    sigma = 0.3
    Sh = (0.3 * rng.standard_normal((n, 2 * nv))).astype(np.float32)
    S = torch.from_numpy(Sh).to(DEV)
    out = torch.zeros_like(S)
    m.predict_seq(S, sigma, out)
    assert torch.count_nonzero(out[:4]) == 0
    ks = range(3, n - 1) if n <= 100 else sorted(set([3, 4, n - 2, *rng.integers(3, n - 1, 60)]))
    for k in ks:
        assert torch.equal(out[k + 1], _one(m, S, int(k), sigma)), k
    P = E.stored_params(params)
    table = L.neighbour_table(rc, nsub)
    for k in (3, n - 2):
        y, _, allow = E.forward(P, E.features_from_slopes(Sh[k::-1][:4], table, sigma))
        ref = Sh[k].astype(np.float64) + sigma * np.concatenate([y[:, 0], y[:, 1]])
        tol = (1e-5 * sigma * np.max(np.abs(y)) + sigma * np.concatenate([allow[:, 0], allow[:, 1]])
               + np.spacing(np.abs(ref).astype(np.float32)))
        assert np.max(np.abs(out[k + 1].cpu().numpy() - ref) / tol) <= 1.0, k


def test_overlapping_output_feeds_back_frame_by_frame():
    m, rc, params, rng = _net(33, 8, 7)
    S = torch.from_numpy((0.3 * rng.standard_normal((12, 66))).astype(np.float32)).to(DEV)
    ref = S.clone()
    for k in range(3, 11):
        ref[k + 1] = _one(m, ref, k, 0.3)
    m.predict_seq(S, 0.3, S)
    assert torch.equal(S, ref)


def test_nan_and_infinite_slopes_stay_local():
    """A NaN slope makes NaN of the predictions that see it in their neighbourhood and
    of no other."""
    m, rc, params, rng = _net(52, 8, 9)
    S = torch.from_numpy((0.3 * rng.standard_normal((9, 104))).astype(np.float32)).to(DEV)
    ref = torch.zeros_like(S)
    m.predict_seq(S, 0.3, ref)
    S[5, 20] = float("nan")
    out = torch.zeros_like(S)
    m.predict_seq(S, 0.3, out)
    sees = (L.neighbour_table(rc, 8) == 20).any(axis=1)
    hit = np.concatenate([sees, sees])
    for k in range(3, 8):
        nan = torch.isnan(out[k + 1]).cpu().numpy()
        want = hit if k >= 5 else np.zeros_like(hit)
        np.testing.assert_array_equal(nan, want)
        keep = torch.from_numpy(~want).to(DEV)
        assert torch.equal(out[k + 1][keep], ref[k + 1][keep])
