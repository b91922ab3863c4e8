"""Shared experts' forward GEMMs in the routed experts' launches against fp64 on the GPU's own
stored inputs: one token, partial and full tiles, shared widths below and above the routed
ones, more shared tiles than routed ones, experts without rows, every tile form."""
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


@pytest.mark.parametrize("pairs", [0, 1, 2])
@pytest.mark.parametrize("rows,d,F,S,Fs", [
    ((1,), 128, 128, 1, 128), ((0, 129, 0), 384, 256, 2, 128), ((100, 157), 256, 128, 3, 1152),
    ((3, 0, 61) * 8, 1152, 384, 8, 256), ((0, 1500, 0, 500), 1024, 1024, 2, 640)])
def test_shared_tiles_follow_the_routed_ones(L, rows, d, F, S, Fs, pairs):
    E, T = len(rows), int(sum(rows))
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    gen = torch.Generator(device="cuda").manual_seed(d + Fs)
    dt = torch.bfloat16
    f = lambda *s: torch.randn(*s, generator=gen, device="cuda")  # noqa: E731
    x, xp = f(T, d).to(dt), f(T, d).to(dt)
    w1, w2 = (0.05 * f(E, 2 * F, d)).to(dt), (0.05 * f(E, d, F)).to(dt)
    ws1, ws2 = (0.05 * f(S, 2 * Fs, d)).to(dt), (0.05 * f(S, d, Fs)).to(dt)
    g = {n: empty(s, dt) for n, s in dict(h=(T, 2 * F), a=(T, F), y=(T, d), hs=(S, T, 2 * Fs), acs=(S, T, Fs),
                                          ys=(S, T, d)).items()}
    cfg = cfg_of(L, mi.MoEShape("f", T, d, E, F, 1, "bf16", n_shared=S, d_ff_shared=Fs))
    L.moe_set_gemm_pairs(pairs)
    try:
        L.moe_expert_ffn_fwd(cfg, xp, dev(off, torch.int32), w1, w2, g["h"], g["a"], g["y"], x, ws1, ws2,
                             g["hs"], g["acs"], g["ys"])
        assert status(L) == 0
    finally:
        L.moe_set_gemm_pairs(2)
    ref = {n: torch.zeros_like(t, dtype=torch.float64) for n, t in g.items()}

    def ffn(xe, w1e, w2e, h, a):
        n = h.shape[1] // 2
        return xe.double() @ w1e.double().T, torch.nn.functional.silu(h[:, :n].double()) * h[:, n:].double(), \
            a.double() @ w2e.double().T
    for e in range(E):
        r = slice(int(off[e]), int(off[e + 1]))
        ref["h"][r], ref["a"][r], ref["y"][r] = ffn(xp[r], w1[e], w2[e], g["h"][r], g["a"][r])
    for i in range(S):
        ref["hs"][i], ref["acs"][i], ref["ys"][i] = ffn(x, ws1[i], ws2[i], g["hs"][i], g["acs"][i])
    for n in ref:
        assert_close(n, g[n], ref[n].cpu().numpy(), TOL["bf16"], stage=True)
