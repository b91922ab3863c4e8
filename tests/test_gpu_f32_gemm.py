"""The fp32 grouped GEMMs (three-way bf16 split on the tensor cores) at the edges of their
tiles and copies: contractions around the 32-term stage, lines
of 4-, 8- and 16-byte alignment, row counts around the 128-row tile, empty experts, one and
several tiles per CTA; operands and sums at both ends of the range, infinities and NaN; an
operand that is aligned to its elements only.

Bound per element of a contraction c = sum a_i b_i: the split leaves out terms below
3 * 2^-25 |a_i b_i|; each of the 12 accumulation steps per 32 terms and each register
addition rounds a partial sum no larger than S = sum |a_i b_i| by at most 2^-23 (truncation),
so |err| <= (12 + K / 32 + 3) * 2^-23 S is a safe worst case."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as mo
from synth import moe_inputs as mi
from tests.gpu_util import cfg_of, dev, empty, need_gpu, status

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return need_gpu()


def close(name, got, ref, mag, K):
    err = np.abs(got.double().cpu().numpy() - ref)
    bound = (16 + K / 32) * 2.0 ** -23 * mag + (2 + K / 32) * 2.0 ** -149
    assert (err <= bound).all(), (name, float((err / bound).max()))


def run(L, rows, d, F, seed, x=None):
    """fwd + bwd of experts with the given row counts; returns buffers and inputs."""
    E, TK = len(rows), int(sum(rows))
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    rng = np.random.default_rng(seed)
    f = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    x = f(TK, d) if x is None else x
    w1, w2, dy = f(E, 2 * F, d) * np.float32(0.1), f(E, d, F) * np.float32(0.1), f(TK, d)
    sh = mi.MoEShape("f", TK, d, E, F, 1, "f32")
    g = {n: empty(s, torch.float32) for n, s in dict(h=(TK, 2 * F), a=(TK, F), y=(TK, d), dh=(TK, 2 * F), dx=(TK, d),
                                                     dw1=(E, 2 * F, d), dw2=(E, d, F)).items()}
    t = {n: dev(v, torch.float32) for n, v in dict(x=x, w1=w1, w2=w2, dy=dy).items()}
    offd = dev(off, torch.int32)
    L.moe_expert_ffn_fwd(cfg_of(L, sh), t["x"], offd, t["w1"], t["w2"], g["h"], g["a"], g["y"])
    L.moe_expert_ffn_bwd(cfg_of(L, sh), t["x"], offd, t["w1"], t["w2"], g["h"], g["a"], t["dy"], g["dh"], g["dx"],
                         g["dw1"], g["dw2"])
    assert status(L) == 0
    return g, off, x, w1, w2, dy


@pytest.mark.parametrize("rows,d,F", [
    ((1, 0, 127, 128, 129), 32, 33),       # 4-byte lines (F odd), one stage, tile edges, an empty expert
    ((31, 32, 33, 63, 64, 65), 64, 62),    # 8-byte lines; weight gradients ending around a stage
    ((5,), 28, 1),                          # less than one stage, one feature
    ((300, 2, 700), 132, 100),              # 16-byte lines, 4 past a stage
    ((2000, 900), 516, 388),                # 128-wide tiles, several per CTA
])
def test_contractions_at_the_edges(L, rows, d, F):
    g, off, x, w1, w2, dy = run(L, rows, d, F, seed=d + F)
    x, w1, w2, dy = (v.astype(np.float64) for v in (x, w1, w2, dy))
    h, a, dh = (g[n].double().cpu().numpy() for n in ("h", "a", "dh"))
    for e in range(len(rows)):
        r = slice(off[e], off[e + 1])
        close("h", g["h"][r], x[r] @ w1[e].T, np.abs(x[r]) @ np.abs(w1[e]).T, d)
        close("y", g["y"][r], a[r] @ w2[e].T, np.abs(a[r]) @ np.abs(w2[e]).T, F)
        close("dx", g["dx"][r], dh[r] @ w1[e], np.abs(dh[r]) @ np.abs(w1[e]), 2 * F)
        close("dw1", g["dw1"][e], dh[r].T @ x[r], np.abs(dh[r]).T @ np.abs(x[r]), rows[e])
        close("dw2", g["dw2"][e], dy[r].T @ a[r], np.abs(dy[r]).T @ np.abs(a[r]), rows[e])
        G, U = h[r, :F], h[r, F:]
        s = mo.sigmoid(G)
        dA, mag = dy[r] @ w2[e], np.abs(dy[r]) @ np.abs(w2[e])
        close("dG", g["dh"][r, :F], dA * U * s * (1 + G * (1 - s)), mag * np.abs(U) * (1 + np.abs(G)), d)
        close("dU", g["dh"][r, F:], dA * G * s, mag * np.abs(G), d)


@pytest.mark.parametrize("xe,we", [(-120, 0), (-140, 10), (-149, 20), (0, -125), (-60, -60), (-100, -50), (60, -128)])
def test_operands_near_the_end_of_the_range(L, xe, we):
    """h = x W1^T with all of x of about 2^xe and all of W1 of about 2^we: the bound above, and
    what the last rounding of an fp32 number that small adds (2^-149 a step: the split's, the
    accumulator's and each register addition's)."""
    rows, d, F = (5, 130), 100, 33
    rng = np.random.default_rng(1000 - xe + we)
    f = lambda e, *s: np.ldexp(rng.standard_normal(s), e).astype(np.float32)  # noqa: E731
    off, x, w1 = np.array([0, 5, 135], np.int32), f(xe, 135, d), f(we, 2, 2 * F, d)
    h, a, y = (empty((135, n), torch.float32) for n in (2 * F, F, d))
    t = lambda v: dev(v, torch.float32)  # noqa: E731
    L.moe_expert_ffn_fwd(cfg_of(L, mi.MoEShape("f", 135, d, 2, F, 1, "f32")), t(x), dev(off, torch.int32), t(w1),
                         t(f(0, 2, d, F)), h, a, y)
    assert status(L) == 0
    for e in range(2):
        r = slice(off[e], off[e + 1])
        xs, ws = x[r].astype(np.float64), w1[e].astype(np.float64)
        err = np.abs(h[r].double().cpu().numpy() - xs @ ws.T)
        bound = (16 + d / 32) * 2.0 ** -23 * (np.abs(xs) @ np.abs(ws).T) + (2 + d / 32) * 2.0 ** -149
        assert (err <= bound).all(), float((err / bound).max())


def test_non_finite_values_follow_ieee(L):
    """A row of x holding an infinity, a NaN or the largest finite value gives what an fp32
    FMA chain gives there, and leaves the other rows alone."""
    rng = np.random.default_rng(3)
    rows, d, F = (40, 90), 96, 70
    x = rng.standard_normal((130, d)).astype(np.float32)
    clean = run(L, rows, d, F, seed=9, x=x.copy())[0]["h"].cpu()
    big = np.float32(3.4028235e38)
    x[3, 5], x[50, 7], x[51, 40], x[129, 95] = np.inf, -np.inf, np.nan, -big
    g, off, _, w1, _, _ = run(L, rows, d, F, seed=9, x=x)
    h = g["h"].cpu()
    assert torch.isinf(h[3]).all() and (torch.sign(h[3]) == torch.sign(torch.from_numpy(w1[0][:, 5]))).all()
    assert torch.isinf(h[50]).all() and (torch.sign(h[50]) == -torch.sign(torch.from_numpy(w1[1][:, 7]))).all()
    assert torch.isnan(h[51]).all()
    want = -big.astype(np.float64) * w1[1][:, 95].astype(np.float64)
    assert np.allclose(h[129].double().numpy(), want, rtol=1e-6, atol=0)
    rest = [i for i in range(130) if i not in (3, 50, 51, 129)]
    assert torch.equal(h[rest], clean[rest])


def test_large_finite_values_follow_the_fma_chain(L):
    """Rows of x whose operands (from 2^105) or sums (from 2^82) leave the split's scaled range:
    what a chain of d FMAs gives, each rounding a partial sum by 2^-24 of it."""
    rows, d, F = (200,), 260, 70
    rng = np.random.default_rng(4)
    f = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    x, w1 = f(200, d), f(1, 2 * F, d) * np.float32(0.1)
    x[3] *= np.float32(1e30)
    x[150:] *= np.float32(2.0 ** 110)
    h, a, y = (empty((200, n), torch.float32) for n in (2 * F, F, d))
    t = lambda v: dev(v, torch.float32)  # noqa: E731
    L.moe_expert_ffn_fwd(cfg_of(L, mi.MoEShape("f", 200, d, 1, F, 1, "f32")), t(x), dev([0, 200], torch.int32), t(w1),
                         t(f(1, d, F)), h, a, y)
    assert status(L) == 0
    x64, w64 = x.astype(np.float64), w1[0].astype(np.float64)
    mag = np.abs(x64) @ np.abs(w64).T
    assert (np.abs(h.double().cpu().numpy() - x64 @ w64.T) <= (16 + d) * 2.0 ** -23 * mag).all()


def test_non_finite_outputs_of_a_long_contraction_wait_as_long_as_they_need(L):
    """One NaN in dY makes dW1 NaN everywhere, a row of dX and of dW2 too: each such output is a
    chain over thousands of rows, during which the other roles wait. Even with a wait limit of
    1 ns the call is right: the repair is no stalled wait (every other wait lasts a few us, and
    a poll sleeps for up to 20)."""
    rows, d, F = (6001, 50), 256, 200
    clean = run(L, rows, d, F, seed=12)[0]
    off = dev([0, 6001, 6051], torch.int32)
    E, TK = 2, 6051
    rng = np.random.default_rng(12)   # the inputs of run()
    f = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    x, w1, w2, dy = f(TK, d), f(E, 2 * F, d) * np.float32(0.1), f(E, d, F) * np.float32(0.1), f(TK, d)
    dy[4000, 7] = np.nan
    t = {n: dev(v, torch.float32) for n, v in dict(x=x, w1=w1, w2=w2, dy=dy).items()}
    dh, dx, dw1, dw2 = (empty(s, torch.float32) for s in ((TK, 2 * F), (TK, d), (E, 2 * F, d), (E, d, F)))
    L.moe_set_wait_limit_ns(1)
    try:
        L.moe_expert_ffn_bwd(cfg_of(L, mi.MoEShape("f", TK, d, E, F, 1, "f32")), t["x"], off, t["w1"], t["w2"],
                             clean["h"], clean["a"], t["dy"], dh, dx, dw1, dw2)
        assert status(L) == 0
    finally:
        L.moe_set_wait_limit_ns(2_000_000_000)
    rest = [i for i in range(TK) if i != 4000]
    assert torch.isnan(dx[4000]).all() and torch.isnan(dw1[0]).all() and torch.isnan(dw2[0, 7]).all()
    assert torch.equal(dx[rest], clean["dx"][rest]) and torch.equal(dw1[1], clean["dw1"][1])
    assert torch.equal(dw2[1], clean["dw2"][1])
    assert torch.equal(dw2[0, [i for i in range(d) if i != 7]], clean["dw2"][0, [i for i in range(d) if i != 7]])


@pytest.mark.parametrize("E", [7, 8, 40])
def test_operand_with_element_alignment(L, E):
    """The router's input gradient with dlogits (the A operand) aligned to one element only,
    beside weights that are copied 16 bytes at a time: pools that leave a contraction tail, so
    that copies of nothing occur in both operands. The same bits as with an aligned dlogits."""
    T, d, k = 150, 132, 2
    rng = np.random.default_rng(E)
    f = lambda *s: dev(rng.standard_normal(s).astype(np.float32), torch.float32)  # noqa: E731
    x, wr, dtw = f(T, d), f(1, E, d), f(T, k)
    pr = torch.softmax(f(T, E), 1)
    w, idx = pr.topk(k, 1)
    cfg = cfg_of(L, mi.MoEShape("r", T, d, E, 128, k, "f32"))
    n = L.moe_workspace_size(cfg)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    got = []
    for shift in (0, 1):
        dl, dx = empty((T * E + 1,), torch.float32)[shift:shift + T * E].view(T, E), empty((T, d), torch.float32)
        assert dl.data_ptr() % 16 == 4 * shift
        L.moe_route_bwd(cfg, x, wr, pr, idx.int(), w.contiguous(), dtw, None, None, dl, empty((1, E, d), torch.float32),
                        empty((1, E), torch.float32), dx, ws, n)
        assert status(L) == 0
        got.append(dx)
        z, wd = dl.double().cpu().numpy(), wr[0].double().cpu().numpy()
        close("dx_router", dx, z @ wd, np.abs(z) @ np.abs(wd), E)
    assert torch.equal(got[0], got[1])
