"""Hidden units far below zero: their GELU vanishes, so they add nothing to the output
however large their outgoing weights are, in the forward pass, the loss and the gradients.

One hidden unit of each layer is pushed to z = -7 .. -60 by its bias and read with a
weight of 1e4.  |GELU| is below 9e-12 from z = -7 on, so the units add less than 1e-7 to
outputs of about one; the tolerance for a network without them is 1e-5 of the largest
output, FP32 arithmetic as in tests/test_gpu_mlp.py.  |GELU'| is below 7e-11, so with
those weights the gradients of their inputs are below 1e-5 of the largest gradient (that
of b3, the mean error)."""
import numpy as np
import pytest
import torch

from synth.mlp_init import flatten, init_mlp_params

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("z", [-7.0, -9.0, -12.0, -20.0, -60.0])
def test_dead_units_add_nothing(z):
    from paper_1805_07254_gb300 import Mlp
    base = {k: np.array(v, np.float32) for k, v in init_mlp_params(3).items()}
    for w in (1, 2):                                 # unit 5 of both layers: no input, a bias
        base[f"W{w}"][5] = 0.0
        base[f"b{w}"][5] = z
    base["W2"][:, 5] = 0.0
    base["W3"][:, 5] = 0.0
    loud = {k: v.copy() for k, v in base.items()}
    loud["W2"][:, 5] = 1e4
    loud["W2"][5] = 0.0
    loud["W3"][:, 5] = 1e4
    rng = np.random.default_rng(4)
    X = torch.from_numpy(rng.standard_normal((70, 200)).astype(np.float32)).to(DEV)
    T = torch.from_numpy(rng.standard_normal((70, 2)).astype(np.float32)).to(DEV)
    out, grad = [], []
    for p in (base, loud):
        m = Mlp(params=flatten(p))
        Y, G = torch.zeros((70, 2), device=DEV), torch.zeros(flatten(p).size, device=DEV)
        m.forward(X, Y)
        m.gradient(X, T, G)
        torch.cuda.synchronize()
        out.append(Y.cpu().numpy())
        grad.append(G.cpu().numpy())
    assert np.max(np.abs(out[0])) > 0.1
    assert np.max(np.abs(out[1] - out[0])) <= 1e-5 * np.max(np.abs(out[0]))
    # W1 row 5 and W2 row 5 of the gradient: GELU' of the dead units
    w1, w2 = grad[1][:64 * 200].reshape(64, 200)[5], grad[1][64 * 200 + 64:][:64 * 64].reshape(64, 64)[5]
    assert np.max(np.abs(w1)) <= 1e-5 * np.max(np.abs(grad[1])) and np.all(np.isfinite(grad[1]))
    assert np.max(np.abs(w2)) <= 1e-5 * np.max(np.abs(grad[1]))

