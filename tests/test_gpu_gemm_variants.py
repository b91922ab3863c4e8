"""Grouped GEMM variants on both sides of the rules that choose them (four or eight epilogue
warps: contractions around 1024, 384 rows a group on average; pair or single-CTA tiles by
rounds, 256- and 128-wide): every result of the expert forward and backward against fp64 on
the GPU's own stored inputs, with the tile form left to the rule and with single-CTA tiles."""
import numpy as np
import pytest
import torch

from synth import moe_inputs as mi
from tests._cmp import TOL, assert_close
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


@pytest.mark.parametrize("pairs", [0, 2])
@pytest.mark.parametrize("rows,d,F", [
    ((1,), 128, 128), ((383, 383), 896, 256), ((300, 468), 1024, 128), ((0, 767, 0), 384, 1024),
    ((1, 1149), 640, 896), ((5, 6, 7, 130) * 16, 1152, 128), ((40,) * 32, 2048, 128)])
def test_variants_agree_with_fp64(L, rows, d, F, pairs):
    E, TK = len(rows), int(sum(rows))
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    gen = torch.Generator(device="cuda").manual_seed(d + F)
    dt = torch.bfloat16
    f = lambda *s: torch.randn(*s, generator=gen, device="cuda")  # noqa: E731
    x, dy = f(TK, d).to(dt), f(TK, d).to(dt)
    w1, w2 = (0.05 * f(E, 2 * F, d)).to(dt), (0.05 * f(E, d, F)).to(dt)
    cfg = cfg_of(L, mi.MoEShape("f", TK, d, E, F, 1, "bf16"))
    g = {n: empty(s, dt) for n, s in dict(h=(TK, 2 * F), a=(TK, F), y=(TK, d), dh=(TK, 2 * F), dx=(TK, d),
                                          dw1=(E, 2 * F, d), dw2=(E, d, F)).items()}
    offd = dev(off, torch.int32)
    L.moe_set_gemm_pairs(pairs)
    try:
        L.moe_expert_ffn_fwd(cfg, x, offd, w1, w2, g["h"], g["a"], g["y"])
        L.moe_expert_ffn_bwd(cfg, x, offd, w1, w2, g["h"], g["a"], dy, g["dh"], g["dx"], g["dw1"], g["dw2"])
        assert status(L) == 0
    finally:
        L.moe_set_gemm_pairs(2)
    ref = {n: torch.zeros_like(t, dtype=torch.float64) for n, t in g.items()}
    h, a, dh = (g[n].double() for n in ("h", "a", "dh"))
    for e in range(E):
        r = slice(int(off[e]), int(off[e + 1]))
        xe, dye, w1e, w2e = x[r].double(), dy[r].double(), w1[e].double(), w2[e].double()
        G, U = h[r, :F], h[r, F:]
        s = torch.sigmoid(G)
        dA = dye @ w2e
        ref["h"][r], ref["a"][r], ref["y"][r] = xe @ w1e.T, G * s * U, a[r] @ w2e.T
        ref["dh"][r] = torch.cat([dA * U * s * (1 + G * (1 - s)), dA * G * s], 1)
        ref["dx"][r], ref["dw1"][e], ref["dw2"][e] = dh[r] @ w1e, dh[r].T @ xe, dye.T @ a[r]
    for n in ref:
        assert_close(n, g[n], ref[n].cpu().numpy(), TOL["bf16"], stage=True)
