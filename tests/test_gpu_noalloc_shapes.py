"""The allocation-free reconstruction over the shapes where its split changes: rows
shared by 1, 2, 7 or 14 warps, one element past each, rows of one and of several
panels, an empty row; one row, rows around the warps and the SMs.

Each thread adds at most 32 products per panel in FP32, then come 5 butterfly and 4 tree
additions, the panels and the integrator: (32 + 1) panels + 11 roundings of 2^-24 of the
sum of magnitudes at most, the tolerance (1.5 x for the products' own rounding)."""
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


def _stored(M, store):
    """Device codes, row scales and the values they stand for (float64)."""
    t = torch.from_numpy(M).to(DEV)
    if store == "f32":
        return t, None, M.astype(np.float64)
    if store in ("bf16", "f16"):
        t = t.to(torch.bfloat16 if store == "bf16" else torch.float16)
        return t, None, t.double().cpu().numpy()
    q, sc = (Q.fp8_row_quantise if store == "fp8" else Q.int8_row_quantise)(M)
    q = torch.from_numpy(np.ascontiguousarray(q))
    codes = q.float().to(torch.float8_e4m3fn) if store == "fp8" else q.to(torch.int8)
    val = np.asarray(q, np.float64) * np.asarray(sc, np.float64)[:, None]
    return codes.to(DEV), torch.from_numpy(sc.astype(np.float32)).to(DEV), val


@pytest.mark.parametrize("store", ["f32", "bf16", "f16", "fp8", "int8"])
@pytest.mark.parametrize("nact,kpad", [(1, 16), (69, 0), (14, 1024), (15, 1040), (151, 2048), (153, 2064), (13, 7168),
                                       (449, 7184), (152, 14336), (40, 14352), (7, 30000), (3000, 160)])
def test_shapes(store, nact, kpad):
    from paper_1805_07254_gb300.rtc import mvm_integrate_noalloc
    rng = np.random.default_rng(nact + kpad)
    M = (rng.standard_normal((nact, kpad)) / max(1, kpad) ** 0.5).astype(np.float32)
    d_M, d_sc, Ms = _stored(M, store) if kpad else (torch.zeros((nact, 16), device=DEV),
                                                    torch.ones(nact, device=DEV), np.zeros((nact, 0)))
    s = (0.3 * rng.standard_normal(kpad)).astype(np.float32)
    d_s = torch.zeros(max(kpad, 16), device=DEV)
    d_s[:kpad] = torch.from_numpy(s)
    a = rng.standard_normal(nact).astype(np.float32)
    ref, mag = Ms @ s.astype(np.float64), np.abs(Ms) @ np.abs(s.astype(np.float64))
    want = float(np.float32(0.99)) * a.astype(np.float64) + float(np.float32(0.4)) * ref
    panels = -(-kpad // 14336)
    tol = 1.5 * (33 * panels + 11) * 2.0 ** -24 * (mag + np.abs(a))
    got = []
    for ksplit in (1, 16):
        d_a = torch.from_numpy(a).to(DEV)
        dm = torch.full((nact + 1,), 5.0, device=DEV)
        mvm_integrate_noalloc(d_M, store, d_sc, nact, kpad, d_s, d_a, dm, 0.4, 0.99, ksplit,
                              stream=torch.cuda.current_stream())
        out = dm.cpu().numpy()
        assert np.all(np.abs(out[:nact] - want) <= tol), np.max(np.abs(out[:nact] - want) / tol)
        assert out[nact] == 5.0 and np.array_equal(d_a.cpu().numpy(), out[:nact])
        got.append(out)
    assert np.array_equal(got[0], got[1])
