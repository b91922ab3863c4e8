"""Router logits and gating on the CUDA cores (fp32, and bf16 pools that are not a multiple
of 4) at the edges: token counts around the 2-, 8- and 16-token groups and the line between
the first two (608), d around the 128-column chunk and the 256-column step, every padded pool
size, clusters of 1 to 8 CTAs per group with uneven column shares, parties of unequal and zero
size. The fp32 sums are compared with 64 bits: chains of at most d / 128 + 32 + 8 additions
(fp32), d / 32 + 8 + 5 (bf16) round each partial sum by 2^-24 of sum |x w|, and picks equal the
oracle's on those logits."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as mo
from synth import moe_inputs as mi
from tests._cmp import assert_close, ints
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


@pytest.mark.parametrize("dtype,T,d,E,k,po", [
    ("f32", 1, 4, 3, 2, None), ("f32", 7, 124, 8, 2, None), ("f32", 9, 132, 9, 3, [0, 0, 5, 9]),
    ("f32", 5000, 260, 17, 4, [0, 4999, 5000]), ("f32", 33, 1000, 64, 8, None),
    ("bf16", 15, 128, 5, 1, None), ("bf16", 17, 256, 13, 3, [0, 9, 9, 17]), ("bf16", 4900, 384, 30, 2, None),
    ("bf16", 500, 2048, 63, 6, [0, 1, 300, 500]),
    ("bf16", 608, 128, 9, 2, [0, 7, 608]), ("bf16", 609, 1280, 25, 4, None), ("bf16", 1, 1152, 63, 6, None), ("bf16", 64, 2048, 33, 6, None), ("bf16", 90, 640, 7, 2, [0, 30, 30, 90]),
    ("f32", 300, 1280, 60, 4, None), ("f32", 40, 900, 8, 2, None), ("f32", 700, 2052, 16, 3, [0, 350, 700])])
def test_route_on_the_cuda_cores(L, dtype, T, d, E, k, po):
    rng = np.random.default_rng(T + d + E)
    rnd = mi.bf16_round if dtype == "bf16" else (lambda a: a)
    P = len(po) - 1 if po else 1
    x = rnd(rng.standard_normal((T, d)).astype(np.float32))
    wr = rnd((rng.standard_normal((P, E, d)) * 0.05).astype(np.float32))
    bias = rng.standard_normal((P, E)).astype(np.float32)
    cut = po or [0, T]
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    sh = mi.MoEShape("r", T, d, E, 128, k, dtype, n_parties=P)
    logits, probs = empty((T, E), torch.float32), empty((T, E), torch.float32)
    idx, w, counts = empty((T, k), torch.int32), empty((T, k), torch.float32), empty((P, E), torch.int32)
    L.moe_route(cfg_of(L, sh), dev(x, dt), dev(wr, dt), dev(bias, torch.float32),
                dev(np.array(po, np.int32), torch.int32) if po else None, logits, probs, idx, w, counts)
    assert status(L) == 0
    z, mag = np.zeros((T, E)), np.zeros((T, E))
    for p in range(P):
        r = slice(cut[p], cut[p + 1])
        z[r] = x[r].astype(np.float64) @ wr[p].astype(np.float64).T + bias[p]
        mag[r] = np.abs(x[r].astype(np.float64)) @ np.abs(wr[p].astype(np.float64)).T + np.abs(bias[p])
    got = logits.double().cpu().numpy()
    terms = d / 128 + 40 if dtype == "f32" else d / 32 + 13
    assert (np.abs(got - z) <= terms * 2.0 ** -24 * mag).all()
    ref = mo.topk_indices(logits.cpu().numpy(), k)
    assert (ints(idx) == ref).all()
    assert (ints(counts) == mo.party_counts(ref, E, np.array(cut, np.int32))).all()
    pr = mo.softmax(got)
    assert_close("probs", probs, pr, 1e-6)
    assert_close("topk_w", w, mo.gate_weights(pr, ref, 0), 1e-6)


@pytest.mark.parametrize("T,d,E", [(5, 128, 5), (40, 3072, 43), (700, 1152, 13), (610, 640, 63)])
def test_bf16_logits_keep_their_order_of_summation(L, T, d, E):
    """Bit for bit: a chain per lane over the 16-byte vectors l, l + 32, ... (a product of two bf16
    values is exact in fp32, so an FMA is one fp32 addition), the 32 chains by a butterfly. An
    order of summation that sums chunks of columns apart is up to a quarter further off 64 bits."""
    rng = np.random.default_rng(T + d)
    x = mi.bf16_round(rng.standard_normal((T, d)).astype(np.float32))
    wr = mi.bf16_round((rng.standard_normal((1, E, d)) * 0.05).astype(np.float32))
    o = [empty((T, E), torch.float32), empty((T, E), torch.float32), empty((T, 1), torch.int32), empty((T, 1), torch.float32),
         empty((1, E), torch.int32)]
    L.moe_route(cfg_of(L, mi.MoEShape("r", T, d, E, 128, 1, "bf16")), dev(x, torch.bfloat16), dev(wr, torch.bfloat16), None,
                None, *o)
    assert status(L) == 0
    steps = -(-d // 256)
    pad = lambda a: np.pad(a, ((0, 0), (0, 256 * steps - d))).reshape(-1, steps, 32, 8)  # noqa: E731
    xs, ws = pad(x), pad(wr[0])
    lane = np.zeros((T, E, 32), np.float32)
    for v in range(steps):
        for q in range(8):
            lane += xs[:, None, v, :, q] * ws[None, :, v, :, q]
    for h in (16, 8, 4, 2, 1):
        lane = lane[..., :h] + lane[..., h:2 * h]
    assert np.array_equal(o[0].cpu().numpy(), lane[..., 0])
