"""The token kernels where their work split changes: dispatch tables at 8 chunks of 128 tokens
and one past (every block counts the picks itself, or the counting kernel runs), pools of 1
to 256 experts in both layouts; gather, combine, its backward and unpermute-reduce with one to
eight warps per token (batch and row sizes around each), every padded number of picks, and
zero to three shared experts. Tables exact; sums against fp64: fp32 accumulation of at most
k + S + 1 terms and one rounding to the storage type."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as mo
from synth import moe_inputs as mi
from tests._cmp import ints
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


def rand_picks(T, E, k, seed):
    r = np.random.default_rng(seed).random((T, E))
    return np.argsort(r, axis=1)[:, :k].astype(np.int32)


@pytest.mark.parametrize("T,E,k,P", [
    (1, 1, 1, 1), (127, 3, 2, 1), (128, 64, 6, 1), (129, 200, 8, 1), (1024, 256, 8, 1), (1025, 33, 5, 1),
    (5000, 64, 6, 1), (9000, 256, 3, 1), (300, 7, 3, 3), (1500, 13, 4, 5), (20000, 100, 2, 2)])
def test_dispatch_tables(L, T, E, k, P):
    idx = rand_picks(T, E, k, T + E)
    sh = mi.MoEShape("t", T, 128, E, 128, k, "bf16", n_parties=P)
    cfg = cfg_of(L, sh)
    x = dev(np.random.default_rng(1).standard_normal((T, 128)), torch.bfloat16)
    off, slot, tok = empty((E + 1,), torch.int32), empty((T * k,), torch.int32), empty((T * k,), torch.int32)
    xp, nb = empty((T * k, 128), torch.bfloat16), L.moe_workspace_size(cfg)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    idxd = dev(idx, torch.int32)
    L.moe_dispatch(cfg, idxd, x, off, slot, tok, xp, ws, nb)
    assert status(L) == 0
    _, ro, rs, rt = mo.dispatch_tables(idx, E)
    assert (ints(off) == ro).all() and (ints(slot) == rs.reshape(-1)).all() and (ints(tok) == rt).all()
    assert torch.equal(xp, x[torch.from_numpy(np.asarray(rt)).long().cuda()])
    if P > 1:
        po = np.linspace(0, T, P + 1).astype(np.int32)
        ge, send = empty((E,), torch.int32), empty((P, P), torch.int32)
        L.moe_dispatch_owner(cfg, idxd, x, dev(po, torch.int32), ge, off, slot, tok, xp, send, ws, nb)
        assert status(L) == 0
        order = sorted(range(E), key=lambda e: (e % P, e))
        assert ints(ge).tolist() == order
        sizes = np.bincount(idx.reshape(-1), minlength=E)
        assert (ints(off) == np.concatenate([[0], np.cumsum(sizes[order])])).all()
        seg = {e: g for g, e in enumerate(order)}
        rows = sorted(((seg[idx[t, j]], t, j) for t in range(T) for j in range(k)))
        want = np.empty(T * k, np.int64)
        for r, (_, t, j) in enumerate(rows):
            want[t * k + j] = r
        assert (ints(slot) == want).all()


@pytest.mark.parametrize("dtype,T,d,k,S", [
    ("bf16", 1, 4096, 1, 0), ("bf16", 9, 128, 2, 1), ("bf16", 64, 2048, 6, 2), ("bf16", 300, 1152, 3, 3),
    ("bf16", 1300, 3072, 5, 0), ("bf16", 2500, 640, 8, 1), ("bf16", 33, 8192, 7, 0),
    ("f32", 3, 4, 2, 0), ("f32", 70, 516, 4, 2), ("f32", 1250, 1000, 6, 1), ("f32", 2600, 132, 1, 0)])
def test_combine_and_unpermute(L, dtype, T, d, k, S):
    rng = np.random.default_rng(T + d + k)
    rnd = mi.bf16_round if dtype == "bf16" else (lambda a: a)
    f = lambda *s: rnd(rng.standard_normal(s).astype(np.float32))  # noqa: E731
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    Fs = 128 if S else 0
    cfg = cfg_of(L, mi.MoEShape("t", T, d, max(k, 2), 128, k, dtype, n_shared=S, d_ff_shared=Fs))
    slot = rng.permutation(T * k).astype(np.int32)
    y, dout, w = f(T * k, d), f(T, d), rng.random((T, k)).astype(np.float32)
    ysh, xr = (f(S, T, d) if S else None), f(T, d)
    out, dx = empty((T, d), dt), empty((T, d), dt)
    dy, dw = empty((T * k, d), dt), empty((T, k), torch.float32)
    yd, sd, wd = dev(y, dt), dev(slot, torch.int32), dev(w, torch.float32)
    shd = dev(ysh, dt) if S else None
    L.moe_combine_fwd(cfg, yd, wd, sd, shd, out)
    L.moe_combine_bwd(cfg, dev(dout, dt), yd, wd, sd, dy, dw)
    L.moe_dispatch_bwd(cfg, yd, sd, dev(xr, dt), shd, dx)
    assert status(L) == 0
    rows = y.astype(np.float64)[slot].reshape(T, k, d)
    w64, g64 = w.astype(np.float64), dout.astype(np.float64)
    sh = ysh.astype(np.float64).sum(0) if S else 0.0
    sha = np.abs(ysh.astype(np.float64)).sum(0) if S else 0.0
    ulp = 2.0 ** -8 if dtype == "bf16" else 2.0 ** -23

    def close(name, got, ref, mag):
        err = np.abs(got.double().cpu().numpy() - ref)
        assert (err <= ulp * np.abs(ref) + (k + S + 2) * 2.0 ** -23 * mag).all(), name

    close("out", out, (w64[:, :, None] * rows).sum(1) + sh, (w64[:, :, None] * np.abs(rows)).sum(1) + sha)
    close("dx", dx, rows.sum(1) + xr + sh, np.abs(rows).sum(1) + np.abs(xr) + sha)
    want = np.empty((T * k, d))
    want[slot] = (w64[:, :, None] * g64[:, None]).reshape(T * k, d)
    close("dy", dy, want, np.abs(want))
    err = np.abs(dw.double().cpu().numpy() - (rows * g64[:, None]).sum(2))
    assert (err <= (d / 8 + 16) * 2.0 ** -24 * (np.abs(rows) * np.abs(g64[:, None])).sum(2)).all()
