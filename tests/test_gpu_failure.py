"""Failure detection on the GPU without faulting it: every mbarrier wait in the
tensor-core kernels is bounded in time. With a 1 ns limit the waits run out, the
kernels record MOE_ERR_TIMEOUT, drain their in-flight copies and MMAs, free TMEM and
return; the same CUDA context then computes correct results again."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as mo
from synth import moe_inputs as mi
from tests._cmp import TOL, assert_close
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status
from tests.test_gpu_dispatch_combine import picks

pytestmark = pytest.mark.gpu


def _ffn_fwd(L, T=512, d=256, E=4, F=256, k=2):
    idx = picks(T, E, k, "uniform", seed=5)
    counts, off, slot, tok = mo.dispatch_tables(idx, E)
    rng = np.random.default_rng(9)
    x = mi.bf16_round(rng.standard_normal((T, d)).astype(np.float32))
    w1 = mi.bf16_round((rng.standard_normal((E, 2 * F, d)) * 0.05).astype(np.float32))
    w2 = mi.bf16_round((rng.standard_normal((E, d, F)) * 0.05).astype(np.float32))
    sh = mi.MoEShape("f", T, d, E, F, k, "bf16")
    cfg = cfg_of(L, sh)
    TK = T * k
    h, a, y = empty((TK, 2 * F), torch.bfloat16), empty((TK, F), torch.bfloat16), empty((TK, d), torch.bfloat16)
    L.moe_expert_ffn_fwd(cfg, dev(x[tok], torch.bfloat16), dev(off, torch.int32), dev(w1, torch.bfloat16),
                         dev(w2, torch.bfloat16), h, a, y)
    ref = np.zeros((TK, d))
    for e in range(E):
        r = slice(off[e], off[e + 1])
        ref[r] = mo.swiglu_forward(x[tok][r], w1[e], w2[e])[3]
    return y, ref


def test_bounded_wait_timeout_is_reported_and_context_survives():
    L = need_gpu()
    assert status(L) == 0
    L.moe_set_wait_limit_ns(1)
    try:
        # a long contraction (d = 8192, 128 k-blocks per tile): the epilogue's wait for
        # the first accumulator lasts tens of microseconds and runs out
        _ffn_fwd(L, T=256, d=8192, E=2, F=256, k=1)
        code = status(L)
    finally:
        L.moe_set_wait_limit_ns(2_000_000_000)
    assert code == L.MOE_ERR_TIMEOUT
    # the context is intact: the same call now succeeds and matches the oracle
    y, ref = _ffn_fwd(L)
    assert status(L) == 0
    assert_close("y", y, ref, TOL["bf16"])


def _router(L, d):
    """bf16 router of a short batch (tiles of 16 tokens whose epilogue warps give up together).
    Tolerance: d / 16 accumulation steps that each truncate a partial sum by up to 2^-23 of it,
    4.9e-4 for d = 65536."""
    T, E, k = 40, 64, 4
    gen = torch.Generator(device="cuda").manual_seed(d)
    x = torch.randn(T, d, generator=gen, device="cuda").bfloat16()
    wr = (torch.randn(1, E, d, generator=gen, device="cuda") * 0.02).bfloat16()
    logits, probs, w = (empty((T, n), torch.float32) for n in (E, E, k))
    idx, counts = empty((T, k), torch.int32), empty((1, E), torch.int32)
    L.moe_route(cfg_of(L, mi.MoEShape("r", T, d, E, 128, k, "bf16")), x, wr, None, None, logits, probs, idx, w, counts)
    return logits, x.double() @ wr[0].double().T, 5e-4


def _pair_weight_gradient(L, rows):
    """bf16 expert backward as CTA pairs; dW1 contracts over an odd number of rows (the last
    k-block is zeroed and credited by the pair's second CTA)."""
    d, F = 256, 256
    gen = torch.Generator(device="cuda").manual_seed(rows)
    f = lambda *s: (torch.randn(*s, generator=gen, device="cuda") * 0.1).bfloat16()  # noqa: E731
    x, dy, h, act, w1, w2 = f(rows, d), f(rows, d), f(rows, 2 * F), f(rows, F), f(1, 2 * F, d), f(1, d, F)
    dh, dx, dw1, dw2 = (empty(s, torch.bfloat16) for s in ((rows, 2 * F), (rows, d), (1, 2 * F, d), (1, d, F)))
    L.moe_set_gemm_pairs(L.MOE_PAIRS_ALL)
    try:
        L.moe_expert_ffn_bwd(cfg_of(L, mi.MoEShape("f", rows, d, 1, F, 1, "bf16")), x, dev([0, rows], torch.int32), w1, w2,
                             h, act, dy, dh, dx, dw1, dw2)
    finally:
        L.moe_set_gemm_pairs(L.MOE_PAIRS_AUTO)
    return dw1[0], dh.double().T @ x.double(), TOL["bf16"]


@pytest.mark.parametrize("call,long,short", [(_router, 65536, 640), (_pair_weight_gradient, 60001, 1111)])
def test_every_kernel_form_gives_up_and_recovers(call, long, short):
    """The short router tiles and the K-variable pairs on a contraction of well over 40 us (a
    wait sleeps up to twice 20 us before it looks at its limit): reported, and the same and a
    shorter call are right afterwards. (No wait of the fp32 GEMM lasts that long: it hands over
    an accumulator every 32 terms.)"""
    L = need_gpu()
    assert status(L) == 0
    L.moe_set_wait_limit_ns(1)
    try:
        call(L, long)
        code = status(L)
    finally:
        L.moe_set_wait_limit_ns(2_000_000_000)
    assert code == L.MOE_ERR_TIMEOUT
    for n in (long, short):
        got, ref, tol = call(L, n)
        assert status(L) == 0
        assert_close(call.__name__, got, ref.cpu().numpy(), tol)
