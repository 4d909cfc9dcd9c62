"""Calls of 2 to 255 tokens (the streaming expert kernels) at the edges of their tiles, against the
CPU oracle: rows and K lengths that are not multiples of the 64-record boxes or the 128-weight
stages, and experts that serve 1, 8, 9, 32, 33 or more assignments."""
import numpy as np
import pytest

import oracle
import synth
from mfharness import Ctx, Payloads, Shape, assert_outputs_close

pytestmark = pytest.mark.gpu

# The kernels keep 24 bits of every operand and sum in fp32: a few roundings of 2^-24 on each of the
# three products of a layer, grown by the sums' lengths (square root of 500 terms at most here), stay
# below 1e-6 of the row in the 2-norm.
REL = 1e-6


@pytest.mark.parametrize("qtype", [synth.Q8_0, synth.Q4_0])
@pytest.mark.parametrize("H,I", [(32, 32), (160, 96), (416, 352), (512, 640)])
def test_stream_tile_edges(qtype, H, I):
    E, k = 12, 3
    shape = Shape(1, H, E, k, I, qtype, model_seed=7)
    ctx = Ctx(shape, E, max_tokens=70)
    pays = Payloads(shape)
    try:
        for T in (2, 8, 9, 32, 33, 70):
            x = synth.activations(T, 0, 0, 0, T, H)
            # expert 0 serves every token, expert 1 all but one, the third choice is spread out
            sets = np.stack([np.zeros(T, int), np.where(np.arange(T) == 1, 2, 1), 3 + np.arange(T) % (E - 3)], 1)
            bias = synth.plant_bias(sets.astype(np.int32), E)
            y, idx, _ = ctx.forward(0, x, bias, T)
            yo, io, _ = oracle.layer(pays.for_layer(0, range(E)), qtype, H, I, k, ctx.wr_host[0], bias, x)
            assert np.array_equal(idx, io)
            assert_outputs_close(y, yo, f"T {T}")
            rel = np.linalg.norm(y - yo, axis=1) / np.linalg.norm(yo, axis=1)
            assert rel.max() <= REL, (T, rel.max())
        assert ctx.mf.mf_check(ctx.h) == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("E,k,slots", [(8, 8, 8), (12, 3, 12), (12, 3, 3)])
@pytest.mark.parametrize("T", [5, 8, 16, 24])
def test_tokens_whose_logits_overflow_leave_the_others_alone(E, k, slots, T):
    """Finite inputs whose router products overflow give logits that are not numbers, and a choice of
    experts that means nothing: the other tokens of the call keep their outputs, and every chosen index is
    an expert.  A stage of the streaming kernels has room for T rounded up to 8 assignments, whatever the
    choice is."""
    H, I = 64, 96
    shape = Shape(1, H, E, k, I, synth.Q8_0, model_seed=11)
    ctx = Ctx(shape, slots, max_tokens=T)
    pays = Payloads(shape)
    try:
        wr = ctx.wr_host[0].copy()
        wr[:, 0] = 4.0
        ctx.wr_host[0] = wr
        ctx.wr[0] = ctx.torch.from_numpy(wr).to(ctx.device)
        x = synth.activations(31, 0, 0, 0, T, H)
        x[:, 0] = 0.0
        good = np.arange(T) % 3 == 1
        x[~good, 0] = 3e38
        y, idx, _ = ctx.forward(0, x, None, T)
        assert ((idx >= 0) & (idx < E)).all()
        yo, io, _ = oracle.layer(pays.for_layer(0, range(E)), synth.Q8_0, H, I, k, wr, None, x[good])
        assert np.array_equal(idx[good], io)
        assert_outputs_close(y[good], yo, f"T {T}")
        assert ctx.mf.mf_check(ctx.h) == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("E,k", [(2, 1), (12, 4)])
def test_calls_of_both_paths_take_turns(E, k):
    """A context of 256 tokens and more keeps the streaming kernels' pieces and the GEMMs' tiles in one
    allocation: calls of both paths, back to back and at every threshold, give the oracle's outputs.  (With two
    experts and top-1 the pieces are the larger.)"""
    H, I, T = 256, 128, 1200
    shape = Shape(1, H, E, k, I, synth.Q8_0, model_seed=17)
    ctx = Ctx(shape, E, max_tokens=T)
    pays = Payloads(shape)
    try:
        x = synth.activations(41, 0, 0, 0, T, H)
        yo, io, _ = oracle.layer(pays.for_layer(0, range(E)), synth.Q8_0, H, I, k, ctx.wr_host[0], None, x)
        torch = ctx.torch
        xd = torch.from_numpy(x).to(ctx.device)
        for threshold in (None, 0, 2, 700, 256):
            if threshold is not None:
                ctx.mf.mf_prefill_threshold(ctx.h, threshold)
            sizes = (T, 255, 256, 3, T, 17, 600)
            ys = [torch.full((n, H), float("nan"), device=ctx.device) for n in sizes]
            for n, y in zip(sizes, ys):
                ctx.mf.mf_moe_forward(ctx.h, 0, xd[:n], ctx.wr[0], None, n, y)
            torch.cuda.synchronize()
            for n, y in zip(sizes, ys):
                assert_outputs_close(y.cpu().numpy(), yo[:n], f"threshold {threshold}, T {n}")
        assert ctx.mf.mf_check(ctx.h) == 0
    finally:
        ctx.close()
