"""Router weight gradients: the reduction of the chunks' partial sums at its edges: one chunk
and more than eight, empty parties, a last block that is part empty, and output counts just
below and above the line between its two forms (150000). Bounds against 64 bits on the
gradients of the logits that the call itself returns: a chunk of at most C tokens adds C terms,
a sum ceil(chunks / 8) of them, the total 8, each rounding by 2^-24 of sum |dz x| (2^-23 for
the tensor cores' accumulation); bf16 results round once more."""
import numpy as np
import pytest
import torch

from synth import moe_inputs as mi
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


@pytest.mark.parametrize("dtype,T,d,E,po", [
    ("f32", 1, 4, 2, None), ("f32", 33, 12, 3, [0, 0, 1, 33]), ("f32", 600, 132, 7, None),
    ("f32", 400, 2340, 64, None), ("f32", 400, 2344, 64, None), ("f32", 333, 1000, 52, [0, 10, 10, 333]),
    ("bf16", 5, 128, 2, None), ("bf16", 3000, 1152, 13, [0, 1, 2000, 3000]), ("bf16", 700, 2560, 60, None),
    ("bf16", 2100, 1152, 63, [0, 2000, 2000, 2100])])
def test_router_gradients_sum_every_chunk(L, dtype, T, d, E, po):
    rng = np.random.default_rng(T + d + E)
    rnd = mi.bf16_round if dtype == "bf16" else (lambda a: a)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    P, k = (len(po) - 1 if po else 1), 2
    cut = po or [0, T]
    x = rnd(rng.standard_normal((T, d)).astype(np.float32))
    wr = rnd((rng.standard_normal((P, E, d)) * 0.05).astype(np.float32))
    pr = np.exp(rng.standard_normal((T, E)))
    pr = (pr / pr.sum(1, keepdims=True)).astype(np.float32)
    idx = np.argsort(-pr, 1)[:, :k].astype(np.int32)
    dw, dbias = empty((P, E, d), dt), empty((P, E), torch.float32)
    dlogits = empty((T, E), torch.float32)
    cfg = cfg_of(L, mi.MoEShape("r", T, d, E, 128, k, dtype, n_parties=P))
    n = L.moe_workspace_size(cfg)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    L.moe_route_bwd(cfg, dev(x, dt), dev(wr, dt), dev(pr, torch.float32), dev(idx, torch.int32),
                    dev(np.take_along_axis(pr, idx, 1), torch.float32),
                    dev(rng.standard_normal((T, k)).astype(np.float32), torch.float32),
                    dev(rng.standard_normal((P, E)).astype(np.float32) * 1e-2, torch.float32),
                    dev(np.array(po, np.int32), torch.int32) if po else None, dlogits, dw, dbias,
                    empty((T, d), dt), ws, n)
    assert status(L) == 0
    dl = dlogits.double().cpu().numpy()
    dz = dlogits.to(dt).double().cpu().numpy()   # the contraction's operand
    got, gotb = dw.double().cpu().numpy(), dbias.double().cpu().numpy()
    x64 = x.astype(np.float64)
    terms = 32 + T / 256 + 10 if dtype == "f32" else 2 * (T + 10)
    for p in range(P):
        r = slice(cut[p], cut[p + 1])
        ref, mag = dz[r].T @ x64[r], np.abs(dz[r]).T @ np.abs(x64[r])
        out = 2.0 ** -8 * np.abs(ref) if dtype == "bf16" else 0.0
        assert (np.abs(got[p] - ref) <= terms * 2.0 ** -24 * mag + out).all()
        bmag = np.abs(dl[r]).sum(0)
        assert (np.abs(gotb[p] - dl[r].sum(0)) <= (T + 10) * 2.0 ** -24 * bmag).all()
