"""Chunks of a cut sequence that the backward joins: whatever pairs are listed, the pairs it works on (as hydra_bwd_bands shows
them, with a scratch that holds everything) cover the same visible positions as often as the listed ones."""
import numpy as np
import pytest

import paper_2609_34318_b200 as P

ROOM = 1 << 40


def counts(cu, pairs, causal):
    """How often each (sequence, q, k) that the mask leaves visible is covered."""
    got = [np.zeros((cu[b + 1] - cu[b],) * 2, dtype=np.int32) for b in range(len(cu) - 1)]
    for p in pairs:
        got[p["seq"]][p["q_start"]:p["q_start"] + p["q_len"], p["k_start"]:p["k_start"] + p["k_len"]] += 1
    return [np.tril(c) if causal else c for c in got]


def listed(rng, cu, drop, extra, cuts_differ):
    """Pairs of sequences cut at random places (q and kv chunks at the same or at other ones), some left out, some added that
    the mask hides altogether."""
    out = []
    for b in range(len(cu) - 1):
        n = int(cu[b + 1] - cu[b])
        cut = lambda: [0] + sorted(set(rng.integers(1, n, size=rng.integers(0, 4)).tolist())) + [n] if n > 1 else [0, n]
        q, k = cut(), cut()
        if not cuts_differ:
            k = q
        for i in range(len(q) - 1):
            for j in range(len(k) - 1):
                visible = k[j] < q[i + 1]
                if visible and rng.random() < drop or not visible and rng.random() >= extra:
                    continue
                out.append((b, q[i], q[i + 1] - q[i], k[j], k[j + 1] - k[j]))
    pairs = np.zeros(len(out), dtype=P.PAIR_DTYPE)
    for i, (b, qs, ql, ks, kl) in enumerate(out):
        pairs[i] = (b, qs, ql, ks, kl, i, 0, 0)
    group, last = -1, None
    for i, o in enumerate(out):
        if o[:3] != last:
            group, last = group + 1, o[:3]
        pairs[i]["group"] = group
    return pairs


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("cuts_differ", [False, True])
@pytest.mark.parametrize("drop,extra", [(0.0, 0.0), (0.0, 0.5), (0.15, 0.0), (0.4, 0.3)])
def test_the_same_positions_are_covered(causal, cuts_differ, drop, extra):
    rng = np.random.default_rng(int(1000 * drop + 10 * extra) + causal + 2 * cuts_differ)
    whole = 0
    for _ in range(25):
        cu = np.concatenate([[0], np.cumsum(rng.integers(1, 300, size=rng.integers(1, 4)))]).astype(np.int32)
        pairs = listed(rng, cu, drop, extra, cuts_differ)
        if not len(pairs):
            continue
        got, _, n_bands = P.hydra_bwd_bands(cu, 2, pairs, causal, ROOM)
        if n_bands == 0:                               # (a pair without visible rows: the backward does not band)
            continue
        assert n_bands == 1
        for a, b in zip(counts(cu, pairs, causal), counts(cu, got, causal)):
            assert np.array_equal(a, b)
        whole += sum(1 for p in got if p["q_len"] == p["k_len"] == cu[p["seq"] + 1] - cu[p["seq"]])
        if drop == 0.0 and causal:                     # nothing is missing: every sequence is one pair again
            assert len(got) == len(cu) - 1
    assert whole > 0


def test_what_is_not_the_whole_triangle_once_stays_as_listed():
    cu = np.array([0, 400], dtype=np.int32)
    pairs, _, _, _ = P.hydra_zigzag_pairs(cu, 2)
    assert len(P.hydra_bwd_bands(cu, 4, pairs, True, ROOM)[0]) == 1
    assert len(P.hydra_bwd_bands(cu, 4, pairs[:-1], True, ROOM)[0]) == len(pairs) - 1
    assert len(P.hydra_bwd_bands(cu, 4, pairs, False, ROOM)[0]) == len(pairs)


def test_the_workspace_holds_either_form():
    for cp_r in (1, 2, 4):
        cu = np.array([0, 900, 1000, 3333], dtype=np.int32)
        pairs, _, _, _ = P.hydra_zigzag_pairs(cu, cp_r)
        for h, hk, d in ((4, 4, 192), (8, 2, 128)):
            cut = P.hydra_workspace_bytes_dims(P.HYDRA_WS_BWD, cu, h, hk, d, 128, pairs)
            assert cut >= P.hydra_workspace_bytes_dims(P.HYDRA_WS_BWD, cu, h, hk, d, 128, None)


def test_the_plan_timer_times_the_tables_that_the_call_builds():
    """Sequences cut in 64 chunks have 2080 pairs each, or one, joined: without a mask all are listed."""
    cu = np.arange(0, 101 * 512, 512, dtype=np.int32)
    pairs, _, _, _ = P.hydra_zigzag_pairs(cu, 32)
    assert P.hydra_plan_describe(P.HYDRA_WS_BWD, cu, 2, pairs=pairs)["pairs"] == 100
    assert P.hydra_plan_describe(P.HYDRA_WS_BWD, cu, 2, pairs=pairs, causal=False)["pairs"] == len(pairs)
    best = lambda causal: min(P.hydra_plan_build_seconds(P.HYDRA_WS_BWD, cu, 2, pairs, causal) for _ in range(5))
    assert 2 * best(True) < best(False)


def test_pairs_in_any_order_are_joined():
    cu = np.array([0, 400, 700, 701], dtype=np.int32)
    pairs, _, _, _ = P.hydra_zigzag_pairs(cu, 2)
    turned = pairs[::-1].copy()
    turned["group"] = pairs["group"].max() - turned["group"]
    for got in (P.hydra_bwd_bands(cu, 4, turned, True, ROOM)[0], P.hydra_bwd_bands(cu, 4, pairs, True, ROOM)[0]):
        assert [(int(p["seq"]), int(p["q_len"]), int(p["k_len"])) for p in got] == [(0, 400, 400), (1, 300, 300), (2, 1, 1)]
