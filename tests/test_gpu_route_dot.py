"""Router logits and gating on the CUDA cores (fp32, and bf16 pools that are not a multiple
of 4) at the edges: token counts around the 8- and 16-token groups, d around the 128-column
chunk, every padded pool size, clusters of 1 to 8 CTAs per group with uneven column shares,
parties of unequal and zero size. The fp32 sums are compared
with 64 bits: chains of at most d / 128 + 32 + 8 additions round each partial sum, so
|dz| <= (d / 128 + 40) 2^-24 sum |x w|, and picks equal the oracle's on those logits."""
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
    ("bf16", 1, 1152, 63, 6, None), ("bf16", 64, 2048, 33, 6, None), ("bf16", 90, 640, 7, 2, [0, 30, 30, 90]),
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
    assert (np.abs(got - z) <= (d / 128 + 40) * 2.0 ** -24 * mag).all()
    ref = mo.topk_indices(logits.cpu().numpy(), k)
    assert (ints(idx) == ref).all()
    assert (ints(counts) == mo.party_counts(ref, E, np.array(cut, np.int32))).all()
    pr = mo.softmax(got)
    assert_close("probs", probs, pr, 1e-6)
    assert_close("topk_w", w, mo.gate_weights(pr, ref, 0), 1e-6)
