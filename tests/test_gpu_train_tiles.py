"""The training kernel at the edges of its tiling: 32-sample tiles (one sample, a
remainder, a whole tile, one more) and batches of more tiles than SMs, whose blocks take
several tiles.

Small batches against the FP64 oracle at the device's rounding points (GRAD_TOL of
tests/test_gpu_mlp.py: FP32 arithmetic, 1e-5 of each tensor's largest entry).  A batch
twice another's size halves dy exactly, so every BF16 rounding is the same and the
gradient is the mean of its halves' up to the FP32 summation order: 1e-5 again."""
import numpy as np
import pytest
import torch

import mlp_emul as E
import synth
from oracle import mlp as L
from synth.mlp_init import flatten, init_mlp_params, unflatten

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _grad(m, X, T):
    g, loss = torch.empty(17154, device=DEV), torch.empty(1, device=DEV)
    m.gradient(X.contiguous(), T.contiguous(), g, loss)
    torch.cuda.synchronize()
    return g.cpu().numpy(), loss.item()


@pytest.mark.parametrize("B", [1, 31, 32, 33])
def test_remainders_match_oracle(B):
    from paper_1805_07254_gb300 import Mlp
    params = init_mlp_params(60 + B)
    rng = np.random.default_rng(B)
    X, T, y, _, ref, loss = E.unique_batch(E.stored_params(params), 0.7 * rng.standard_normal((B, 200)),
                                           0.2 * rng.standard_normal((B, 2)), rng)
    m = Mlp(params=flatten(params))
    g, l = _grad(m, torch.from_numpy(X).to(DEV), torch.from_numpy(T).to(DEV))
    errs = {k: E.max_rel(v, ref[k]) for k, v in unflatten(g).items()}
    assert max(errs.values()) <= TOL, errs
    assert abs(l - loss) <= TOL * loss
    Y = torch.full((B + 1, 2), 7.0, device=DEV)
    m.forward(torch.from_numpy(X).to(DEV), Y)
    assert E.max_rel(Y[:B].cpu().numpy(), y) <= TOL and torch.all(Y[B] == 7.0)


def test_blocks_with_several_tiles():
    from paper_1805_07254_gb300 import Mlp
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    half = 32 * sms - 16                      # odd tile counts; twice it is ~2 tiles a block
    gen = torch.Generator(device="cuda").manual_seed(3)
    X = 0.7 * torch.randn((2 * half, 200), generator=gen, device=DEV)
    T = 0.2 * torch.randn((2 * half, 2), generator=gen, device=DEV)
    m = Mlp(params=flatten(init_mlp_params(3)))
    whole, lw = _grad(m, X, T)
    a, la = _grad(m, X[:half], T[:half])
    b, lb = _grad(m, X[half:], T[half:])
    ref = unflatten(0.5 * (a.astype(np.float64) + b))
    errs = {k: E.max_rel(v, ref[k]) for k, v in unflatten(whole).items()}
    assert max(errs.values()) <= TOL, errs
    assert abs(lw - 0.5 * (la + lb)) <= TOL * lw


@pytest.mark.parametrize("B", [33, 5000])
def test_sequence_batches_equal_explicit_ones(B):
    """Samples outside the sequence or the pupil included: zero features and target."""
    from paper_1805_07254_gb300 import Mlp
    cfg = synth.tiny_scao()
    sa, nv, n = cfg.subaps, cfg.n_valid, 25
    rng = np.random.default_rng(B)
    S = (0.3 * rng.standard_normal((n, 2 * nv))).astype(np.float32)
    smp = np.stack([rng.integers(-1, nv + 1, B), rng.integers(2, n, B)], axis=1).astype(np.int32)
    ok = (smp[:, 0] >= 0) & (smp[:, 0] < nv) & (smp[:, 1] >= 3) & (smp[:, 1] <= n - 2)
    table = L.neighbour_table(sa, cfg.nsub)
    X, T = np.zeros((B, 200), np.float32), np.zeros((B, 2), np.float32)
    feats = {k: L.gather_features_table(S[k::-1][:4], table, 1.0) for k in range(3, n - 1)}
    for s in np.flatnonzero(ok):
        i, k = smp[s]
        X[s] = feats[k][i]
        T[s] = (S[k + 1] - S[k])[[i, nv + i]]
    params = flatten(init_mlp_params(8))
    a, b = Mlp(params=params), Mlp(params=params)
    b.set_geometry(sa, cfg.nsub)
    la, lb = torch.empty(1, device=DEV), torch.empty(1, device=DEV)
    dX, dT = torch.from_numpy(X).to(DEV), torch.from_numpy(T).to(DEV)
    dS, dsmp = torch.from_numpy(S).to(DEV), torch.from_numpy(smp).to(DEV)
    for _ in range(3):
        a.train_step(dX, dT, 1e-3, la)
        b.train_seq(dS, dsmp, 1.0, 1e-3, lb)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a.get_params(), b.get_params())
    assert la.item() == lb.item()
