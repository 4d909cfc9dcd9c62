"""The all-at-once form of the slot replacement that calls with several tokens use where its condition
holds (csrc/mf_resolve.cu, lru_parallel): the rule restated on the CPU and compared with the oracle's
access-by-access cache over random calls (whenever the condition accepts a call, hits, slots,
evictions and the state left behind are the oracle's), and the kernel itself on the same calls, of
which some take the rule and some the ordered walk."""
import random

import numpy as np
import pytest

import oracle


def all_at_once(S, expert_of, last, clock, experts):
    """(slots, hits) of the call's distinct experts, or None where the condition does not hold; the
    state (expert_of, last) is updated in place."""
    slot_of = {e: s for s, e in enumerate(expert_of) if e >= 0}
    own = [slot_of.get(e, -1) for e in experts]
    misses_before = np.concatenate([[0], np.cumsum([o < 0 for o in own])]).astype(int)
    n_miss = int(misses_before[-1])
    occ = sorted((s for s in range(S) if expert_of[s] >= 0), key=lambda s: (last[s], s))
    free = [s for s in range(S) if expert_of[s] < 0]
    rank = {s: r for r, s in enumerate(occ)}
    hit_slots = set(s for s in own if s >= 0)
    if n_miss:
        for u, s in enumerate(own):
            if s >= 0:
                older = sum(1 for v in range(u) if own[v] >= 0 and rank[own[v]] < rank[s])
                if max(0, misses_before[u] - len(free)) > rank[s] - older:
                    return None
    base = free + [s for s in occ if s not in hit_slots]
    F = len(base)
    slots = []
    for u, s in enumerate(own):
        m = misses_before[u]
        if s < 0:
            while m >= F:
                v = m - F
                assert v < u
                if own[v] >= 0:
                    s = own[v]
                    break
                m = misses_before[v]
            if s < 0:
                s = base[m]
        slots.append(s)
    for u, (e, s) in enumerate(zip(experts, slots)):
        if F + u >= n_miss:
            expert_of[s], last[s] = e, clock + u + 1
    return slots, [s >= 0 for s in own]


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("E,S,k", [(12, 3, 2), (16, 8, 4), (24, 24, 3), (40, 17, 8), (9, 1, 1)])
def test_all_at_once_replacement_matches_the_oracle(E, S, k, order):
    rng = random.Random(E * 100 + S * 10 + order)
    lru = oracle.LRU(E, S, 1)
    expert_of, last, clock = [-1] * S, [0] * S, 0
    accepted = 0
    for call in range(300):
        T = rng.choice((2, 3, 5, 12))
        hot = rng.randint(k, E)
        idx = np.array([rng.sample(range(hot), k) for _ in range(T)], np.int32)
        experts, slots, hits = (list(map(int, v)) for v in lru.step(idx, order))
        got = all_at_once(S, expert_of, last, clock, experts)
        if got is not None:
            accepted += 1
            assert got == (slots, [bool(h) for h in hits]), call
        else:  # the oracle's decisions, access by access
            for u, (e, s) in enumerate(zip(experts, slots)):
                expert_of[s], last[s] = e, clock + u + 1
        clock += len(experts)
        assert len(set(e for e in expert_of if e >= 0)) == sum(e >= 0 for e in expert_of)
    assert accepted >= (250 if order else 20)


@pytest.mark.gpu
@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("E,S,k", [(12, 3, 2), (16, 8, 4), (24, 24, 3), (40, 17, 8), (9, 1, 1)])
def test_kernel_takes_the_oracles_decisions(E, S, k, order):
    """The same calls through mf_moe_forward: every access (expert, slot, hit), the counters and the
    outputs (each wave's experts in the slots that the record names).  With S experts of E resident and
    first-occurrence order, some calls are refused by the rule and walked in order."""
    import synth
    from mfharness import Ctx, Payloads, Shape, assert_outputs_close, oracle_trace, stats_tuple
    H = I = 32
    rng = random.Random(E * 100 + S * 10 + order)
    shape = Shape(1, H, E, k, I, synth.Q8_0, model_seed=18)
    lru = oracle.LRU(E, S, synth.payload_bytes(H, I, synth.Q8_0))
    ctx = Ctx(shape, S, max_tokens=12)
    pays = Payloads(shape)
    expert_of, last, clock, by_rule, walked = [-1] * S, [0] * S, 0, 0, 0
    try:
        ctx.mf.mf_access_order(ctx.h, order)
        for call in range(150):
            T = rng.choice((2, 3, 5, 12))
            hot = rng.randint(k, E)
            idx = np.array([rng.sample(range(hot), k) for _ in range(T)], np.int32)
            x, bias = synth.activations(51, 0, 0, call, T, H), synth.plant_bias(idx, E)
            y, got, _, trace = ctx.forward(0, x, bias, T, trace=True)
            yo, want, _ = oracle.layer(pays.for_layer(0, range(E)), synth.Q8_0, H, I, k, ctx.wr_host[0], bias, x)
            assert np.array_equal(got, want), call
            assert_outputs_close(y, yo, f"call {call}")
            experts, slots, hits = oracle_trace(lru, got, order)
            assert trace == (experts, slots, hits), call
            if all_at_once(S, expert_of, last, clock, experts) is None:
                walked += 1
                for u, (e, s) in enumerate(zip(experts, slots)):
                    expert_of[s], last[s] = e, clock + u + 1
            else:
                by_rule += 1
            clock += len(experts)
        assert stats_tuple(ctx.mf.mf_stats(ctx.h, 0)) == stats_tuple(lru.stats())
        assert ctx.mf.mf_check(ctx.h) == 0
        assert by_rule > 20 and (walked > 20) == (order == 0 and S < E)
    finally:
        ctx.close()
