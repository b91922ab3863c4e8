"""SGD update at its edges: a single vector, sizes around one and two vectors a thread of the whole
grid, odd sizes and unaligned tensors (one element at a time), groups that were not called,
with and without a master copy. One fused multiply-add per weight: fp32 results within one
rounding (2^-24 of the terms), bf16 weights are the rounded master (or within 2^-8 of the sum, half a
spacing of 8 significant bits)."""
import pytest
import torch

from tests.gpu_util import dev, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


@pytest.mark.parametrize("master", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("G,n,shift", [(1, 1, 0), (3, 8, 0), (2, 7, 0), (1, 2490368 - 8, 0), (1, 2490368 + 8, 0),
                                       (2, 1245184 * 2 + 24, 0), (64, 40960, 0), (3, 4096, 1)])
def test_update_touches_every_weight_once(L, dtype, G, n, shift, master):
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(n + G)
    f = lambda: torch.randn(G * n + shift, generator=gen, device="cuda")  # noqa: E731
    m = f()[shift:]
    w, dw = torch.empty(G * n + shift, dtype=dt, device="cuda")[shift:], f().to(dt)[shift:]
    w.copy_(m)
    called = [(i % 3) != 1 for i in range(G)]
    counts = dev([int(c) for c in called], torch.int32)
    old, base = w.clone(), (m if master else w).double().view(G, n)
    lr = 0.37
    L.moe_sgd_update(w, dw, G, n, counts, lr, L.MOE_F32 if dtype == "f32" else L.MOE_BF16, m if master else None)
    assert status(L) == 0
    step = torch.tensor(lr, dtype=torch.float32).double().item() * dw.double().view(G, n)
    ref, mag = base - step, base.abs() + step.abs()
    got = (m if master else w).double().view(G, n)
    eps = 2.0 ** -8 if dtype == "bf16" and not master else 2.0 ** -24
    for i in range(G):
        if called[i]:
            assert ((got[i] - ref[i]).abs() <= 1.01 * eps * mag[i]).all()
            if master:
                assert torch.equal(w.view(G, n)[i], m.view(G, n)[i].to(dt))
        else:
            assert torch.equal(w.view(G, n)[i], old.view(G, n)[i])
