"""The last tile of an expert in the CTA-pair GEMMs (1 to 128 rows: operands exchanged, rows
as the MMA's N dimension) against fp64 on the GPU's own stored inputs: row counts around every
step of 16, around the 32-row copy boxes and the 128-row limit, alone and behind full tiles;
d and F of 128 mod 256 (a last column tile of one CTA)."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as mo
from synth import moe_inputs as mi
from tests._cmp import TOL, assert_close
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


@pytest.mark.parametrize("rows,d,F", [
    ((1, 2, 15, 16, 17, 31, 32, 33, 63, 64, 65), 256, 384),
    ((127, 128, 129, 0, 255, 256, 257, 272), 384, 128),
    ((256 + 48, 512 + 7, 768 + 100), 2048, 640)])
def test_last_tiles_of_experts(L, rows, d, F):
    E, TK = len(rows), int(sum(rows))
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    rng = np.random.default_rng(d + F)
    f = lambda *s: mi.bf16_round(rng.standard_normal(s).astype(np.float32))  # noqa: E731
    x, w1, w2, dy = f(TK, d), mi.bf16_round(f(E, 2 * F, d) * np.float32(0.05)), mi.bf16_round(f(E, d, F) * np.float32(0.05)), f(TK, d)
    cfg = cfg_of(L, mi.MoEShape("f", TK, d, E, F, 1, "bf16"))
    dt = torch.bfloat16
    g = {n: empty(s, dt) for n, s in dict(h=(TK, 2 * F), a=(TK, F), y=(TK, d), dh=(TK, 2 * F), dx=(TK, d),
                                          dw1=(E, 2 * F, d), dw2=(E, d, F)).items()}
    xd, w1d, w2d, dyd, offd = dev(x, dt), dev(w1, dt), dev(w2, dt), dev(dy, dt), dev(off, torch.int32)
    L.moe_set_gemm_pairs(1)
    try:
        L.moe_expert_ffn_fwd(cfg, xd, offd, w1d, w2d, g["h"], g["a"], g["y"])
        L.moe_expert_ffn_bwd(cfg, xd, offd, w1d, w2d, g["h"], g["a"], dyd, g["dh"], g["dx"], g["dw1"], g["dw2"])
        assert status(L) == 0
    finally:
        L.moe_set_gemm_pairs(2)
    h, a, dh = (g[n].double().cpu().numpy() for n in ("h", "a", "dh"))
    ref = {n: np.zeros((TK, c)) for n, c in dict(y=d, dh=2 * F, dx=d).items()}
    for e in range(E):
        r = slice(off[e], off[e + 1])
        G, U = h[r, :F], h[r, F:]
        s = mo.sigmoid(G)
        dA = dy[r].astype(np.float64) @ w2[e].astype(np.float64)
        ref["y"][r] = a[r] @ w2[e].astype(np.float64).T
        ref["dh"][r] = np.concatenate([dA * U * s * (1 + G * (1 - s)), dA * G * s], 1)
        ref["dx"][r] = dh[r] @ w1[e].astype(np.float64)
    for n in ref:
        assert_close(n, g[n], ref[n], TOL["bf16"], stage=True)
