"""Router of many-token calls (the tiled path, T >= 16) vs the oracle router, through the C ABI.

Real routing (no planted bias) on seeded x and W_r, so the k-th and (k+1)-th logits are often
close: routed indices must equal the oracle's exactly, weights within G_ATOL.  The shapes cover
ragged token tiles (T not a multiple of 32), ragged expert tiles (E not a multiple of 64), one
and many K splits, the smallest and largest expert counts, exact ties at the selection boundary
(identical W_r rows and bias: the lower expert id first), and the switch between the
one-token-per-cluster router (T = 15) and the tiled one (T = 16) on the same tokens."""
import numpy as np
import pytest

import oracle
import synth
from mfharness import Ctx, G_ATOL, Shape

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _check_routes(ctx, x, bias, T, k):
    _, idx, w = ctx.forward(0, x, bias, T)
    for t in range(T):
        _, oidx, og = oracle.router(x[t], ctx.wr_host[0], None if bias is None else bias[t], k)
        assert np.array_equal(idx[t], oidx), (t, idx[t], oidx)
        assert np.abs(w[t] - og).max() <= G_ATOL, t
    return idx


@pytest.mark.parametrize("H,E,k,T", [
    (2048, 100, 8, 300),   # ragged expert tile (64 + 36), 10 token tiles, 16 K splits
    (2048, 128, 8, 4096),  # the 48-layer prefill call: 256 tiles, no K split
    (256, 64, 4, 17),      # one token past a tile edge
    (96, 12, 3, 16),       # fewer experts than a tile, 3 K splits of one chunk
    (64, 1024, 8, 40),     # the largest expert count
    (2816, 128, 8, 64),    # the 30-layer batch-64 shape
])
def test_tiled_router_real_routing(H, E, k, T):
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=5)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        x = synth.activations(21, 0, 0, 0, T, H)
        _check_routes(ctx, x, None, T, k)
        assert ctx.mf.mf_check(ctx.h) == 0
    finally:
        ctx.close()


def test_tiled_router_exact_ties():
    """Rows 5 and 9 of W_r equal and both lifted by the same bias: they lead with equal logits
    (5 before 9); rows 3 and 20 equal with a smaller lift: they tie for the last place (3 wins)."""
    H, E, k, T = 256, 64, 3, 33
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=6)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        import torch
        wr = ctx.wr_host[0].copy()
        wr[9] = wr[5]
        wr[20] = wr[3]
        ctx.wr_host[0] = wr
        ctx.wr[0] = torch.from_numpy(wr).to(ctx.device)
        x = synth.activations(22, 0, 0, 0, T, H)
        bias = np.zeros((T, E), np.float32)
        bias[:, [5, 9]] = 1000.0
        bias[:, [3, 20]] = 500.0
        idx = _check_routes(ctx, x, bias, T, k)
        assert (idx[:, 0] == 5).all() and (idx[:, 1] == 9).all() and (idx[:, 2] == 3).all()
    finally:
        ctx.close()


def test_router_paths_agree_at_the_switch():
    """The same 15 tokens through the per-token router (T = 15) and, with one more token, the
    tiled router (T = 16): identical indices and weights for the 15."""
    H, E, k = 2048, 128, 8
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=7)
    ctx = Ctx(shape, slots=E, max_tokens=16)
    try:
        x = synth.activations(23, 0, 0, 0, 16, H)
        i15 = _check_routes(ctx, x[:15], None, 15, k)
        _, w15 = ctx.forward(0, x[:15], None, 15)[1:]
        i16 = _check_routes(ctx, x, None, 16, k)
        _, w16 = ctx.forward(0, x, None, 16)[1:]
        assert np.array_equal(i15, i16[:15])
        assert np.array_equal(w15, w16[:15])
    finally:
        ctx.close()


@pytest.mark.parametrize("E,T", [(40, 16), (128, 65), (200, 33)])
def test_tiled_router_orders_logits_that_fp32_sums_cannot(E, T):
    """Router rows that differ from one another by a few units in the last place of a few weights: the
    logits agree to more digits than a plain fp32 sum of 1024 products keeps, so only the compensated
    dot product orders them as the oracle does."""
    H, k = 1024, 5
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=9)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        rng = np.random.default_rng(E)
        w = np.tile(ctx.wr_host[0][:1], (E, 1))
        for e in range(1, E):  # 3 of the weights one to four units in the last place away
            at = rng.integers(0, H, 3)
            w[e, at] = (w[e, at].view(np.int32) + rng.integers(-4, 5, 3).astype(np.int32)).view(np.float32)
        ctx.wr_host[0] = w
        ctx.wr[0] = ctx.torch.from_numpy(w).to(ctx.device)
        _check_routes(ctx, synth.activations(23, 0, 0, 0, T, H), None, T, k)
    finally:
        ctx.close()


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("T", [1, 5, 20])
def test_indices_and_weights_reach_any_buffer(T, off):
    """The router stores idx and w itself where the caller's buffers are aligned to their values; buffers
    at an odd address (off = 1) are copied to.  Either one alone, and neighbouring bytes left as they were."""
    H, E, k = 256, 40, 5
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=10)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        torch, n = ctx.torch, T * k * 4
        xh = synth.activations(24, 0, 0, 0, T, H)
        x, y = torch.from_numpy(xh).to(ctx.device), torch.empty(T, H, device=ctx.device)
        for want_i, want_w in ((True, True), (True, False), (False, True)):
            bufs = [torch.full((n + 16,), 0xA5, dtype=torch.uint8, device=ctx.device) for _ in range(2)]
            at = [b.data_ptr() + off if want else None for b, want in zip(bufs, (want_i, want_w))]
            ctx.mf.mf_moe_forward(ctx.h, 0, x, ctx.wr[0], None, T, y, at[0], at[1])
            torch.cuda.synchronize()
            raw = [b.cpu().numpy() for b in bufs]
            for r, want in zip(raw, (want_i, want_w)):
                assert (r[:off] == 0xA5).all() and (r[off + n if want else 0:] == 0xA5).all()
            idx = raw[0][off:off + n].copy().view(np.int32).reshape(T, k)
            w = raw[1][off:off + n].copy().view(np.float32).reshape(T, k)
            for t in range(T):
                _, oidx, og = oracle.router(xh[t], ctx.wr_host[0], None, k)
                assert not want_i or np.array_equal(idx[t], oidx), t
                assert not want_w or np.abs(w[t] - og).max() <= G_ATOL, t
    finally:
        ctx.close()


@pytest.mark.parametrize("E,k,n_nan", [(40, 5, 40), (40, 5, 38), (8, 8, 3), (200, 8, 200)])
@pytest.mark.parametrize("T", [1, 5, 20])
def test_logits_that_are_not_numbers_rank_last(T, E, k, n_nan):
    """Finite inputs whose products overflow (x[0] times four of column 0) give logits that are not
    numbers: they rank after every other, among themselves the lower expert first, so a token's k experts
    are distinct and the same on every call; tokens with x[0] = 0 route as the oracle says."""
    H = 256
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=12)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        bad = np.sort(np.random.default_rng(E + k).permutation(E)[:n_nan])
        fine = np.setdiff1d(np.arange(E), bad)
        wr = ctx.wr_host[0].copy()
        wr[:, 0] = 0.0
        wr[bad, 0] = 4.0
        ctx.wr_host[0] = wr
        ctx.wr[0] = ctx.torch.from_numpy(wr).to(ctx.device)
        x = synth.activations(25, 0, 0, 0, T, H)
        x[:, 0] = 0.0
        x[::2, 0] = 3e38
        _, idx, w = ctx.forward(0, x, None, T)
        for t in range(T):
            if t % 2 == 0:
                z = wr[fine].astype(np.float64) @ x[t].astype(np.float64)
                order = fine[np.lexsort((fine, -z.astype(np.float32)))]
                assert np.array_equal(idx[t], np.concatenate([order, bad])[:k]), t
            else:
                _, oidx, og = oracle.router(x[t], wr, None, k)
                assert np.array_equal(idx[t], oidx) and np.abs(w[t] - og).max() <= G_ATOL, t
    finally:
        ctx.close()


@pytest.mark.parametrize("x_exp,w_exp", [(0, 0), (-80, 0), (0, -75), (-66, -10), (-80, -8), (60, 40)])
def test_tiled_router_orders_cancelling_logits_at_any_scale(x_exp, w_exp):
    """Rows of W_r a few units in the last place apart, x nearly orthogonal to them all, both scaled by
    powers of two (exact): the squares of such values underflow at the small scales, the logits do not,
    and their order is the oracle's at every scale."""
    H, E, k, T = 1024, 40, 5, 48
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=13)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        rng = np.random.default_rng(3)
        w = np.tile(ctx.wr_host[0][:1], (E, 1))
        for e in range(1, E):
            at = rng.integers(0, H, 3)
            w[e, at] = (w[e, at].view(np.int32) + rng.integers(-4, 5, 3).astype(np.int32)).view(np.float32)
        x = synth.activations(26, 0, 0, 0, T, H).astype(np.float64)
        w0 = w[0].astype(np.float64)
        x = (x - np.outer(x @ w0, w0) / (w0 @ w0)).astype(np.float32)
        w = np.ldexp(w, w_exp)
        ctx.wr_host[0] = w
        ctx.wr[0] = ctx.torch.from_numpy(w).to(ctx.device)
        _check_routes(ctx, np.ldexp(x, x_exp), None, T, k)
    finally:
        ctx.close()


@pytest.mark.parametrize("E,k,T", [(8, 8, 16), (40, 5, 33), (128, 8, 65)])
def test_tiled_router_zero_tokens_and_masked_experts(E, k, T):
    """Tokens that are all zero (padding) have their biases as logits, and experts masked by a bias of
    -infinity rank behind all others, the lower first: with and without a bias, beside ordinary tokens."""
    H = 256
    shape = Shape(1, H, E, k, 64, synth.Q8_0, model_seed=14)
    ctx = Ctx(shape, slots=E, max_tokens=T)
    try:
        x = synth.activations(27, 0, 0, 0, T, H)
        x[::3] = 0.0
        x[3::6] = -0.0
        idx = _check_routes(ctx, x, None, T, k)
        assert (idx[::3] == np.arange(k)).all()
        rng = np.random.default_rng(4)
        bias = rng.integers(-2, 3, (T, E)).astype(np.float32)  # ties
        _check_routes(ctx, x, bias, T, k)
        bias[:, rng.permutation(E)[:E - k]] = -np.inf  # k left
        _check_routes(ctx, x, bias, T, k)
        if E > k:  # fewer than k left: the masked experts of the lowest index follow, with weight 0
            bias[:, np.flatnonzero(bias[0] > -np.inf)[:2]] = -np.inf
            _check_routes(ctx, x, bias, T, k)
    finally:
        ctx.close()
