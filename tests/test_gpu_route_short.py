"""Short router tiles (up to 32 tokens, eight lanes a token) against the general form, which
the same tokens take inside a batch of 9999: logits, probabilities and gates equal bit for bit,
picks and counts equal, with equal logits, infinities, the type's lowest value and NaN among
them. Every padded pool size, d that
fills 2 to 64 k-blocks (the last copy part empty), parties that end inside a tile, T around
the limits of both tile heights (16 x 152, 32 x 152)."""
import numpy as np
import pytest
import torch

from synth import moe_inputs as mi
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


def route(L, x, wr, bias, po, E, k, norm):
    T, d = x.shape
    P = len(po) - 1
    sh = mi.MoEShape("r", T, d, E, 128, k, "bf16", n_parties=P, normalize_topk=norm)
    o = [empty((T, E), torch.float32), empty((T, E), torch.float32), empty((T, k), torch.int32),
         empty((T, k), torch.float32), empty((P, E), torch.int32)]
    L.moe_route(cfg_of(L, sh), x, wr, bias, dev(np.array(po, np.int32), torch.int32) if P > 1 else None, *o)
    assert status(L) == 0
    return o


@pytest.mark.parametrize("T,d,E,k,po,norm,odd", [
    (1, 128, 4, 1, None, 0, False), (15, 256, 16, 2, None, 1, True), (33, 4096, 8, 2, None, 0, False),
    (64, 2048, 64, 6, None, 0, True), (100, 640, 32, 8, [0, 0, 37, 100], 1, True), (90, 384, 20, 3, [0, 1, 90], 0, False),
    (2432, 128, 64, 8, None, 1, True), (2433, 1152, 60, 4, [0, 2000, 2433], 0, True), (3000, 256, 12, 2, None, 0, False),
    (4864, 384, 28, 5, None, 1, True), (4865, 128, 16, 16, None, 0, True)])
def test_short_tiles_equal_the_general_form(L, T, d, E, k, po, norm, odd):
    k = min(k, 8)
    gen = torch.Generator(device="cuda").manual_seed(T + d + E)
    po = po or [0, T]
    P, pad = len(po) - 1, 9999 - T
    x = torch.randn(T, d, generator=gen, device="cuda").bfloat16()
    wr = (torch.randn(P, E, d, generator=gen, device="cuda") * 0.05).bfloat16()
    wr[:, E // 2] = wr[:, 0]  # equal logits
    bias = torch.randn(P, E, generator=gen, device="cuda")
    bias[:, E // 2] = bias[:, 0]
    if odd:
        for i, v in enumerate([float("inf"), float("nan"), -float("inf"), torch.finfo(torch.float32).min]):
            bias[i % P, (3 * i + 1) % E] = v
    short = route(L, x, wr, bias, po, E, k, norm)
    # the same tokens, each party padded (the last by whole tiles), in one long batch
    rows = torch.cat([torch.arange(po[p], po[p + 1], device="cuda") for p in range(P)])
    extra = torch.randn(pad, d, generator=gen, device="cuda").bfloat16()
    long_po = po[:-1] + [9999]
    ref = route(L, torch.cat([x, extra]), wr, bias, long_po, E, k, norm)
    assert torch.equal(short[0].view(torch.int32), ref[0][rows].view(torch.int32))
    assert torch.equal(short[2], ref[2][rows])
    for i in (1, 3):
        torch.testing.assert_close(short[i], ref[i][rows], rtol=0, atol=0, equal_nan=True)
    for p in range(P):
        n = torch.bincount(short[2][po[p]:po[p + 1]].flatten().long(), minlength=E)
        assert torch.equal(n, short[4][p].long())
