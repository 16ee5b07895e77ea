"""Work tables of the short-sequence forward, looked at on the host: every row of every pair and head goes to that pair's own
output row once, whether its tile is the pair's alone or shared with other pairs, wherever its table entry lies."""
import numpy as np
import pytest

import paper_2609_34318_b200 as P

ITEM = np.dtype([("q_tok0", "<i4"), ("k_tok0", "<i4"), ("k_len", "<i4"), ("off", "<i4"), ("out_row0", "<i4"), ("head", "<u2"),
                 ("n_kv", "<u2"), ("rows", "u1"), ("to_part", "u1"), ("half", "u1"), ("n_segs", "u1"), ("first_seg", "<u4")])
SEG = np.dtype([("begin", "<i2"), ("to_part", "<i2"), ("delta", "<i4")])


@pytest.fixture
def all_pairs_short():
    P.hydra_set_fwd_short_len(1 << 21)
    yield
    P.hydra_set_fwd_short_len(-1)


def tables(cu, h, pairs, causal=True, h_kv=None, d_qk=192):
    plan, raw = P.hydra_plan_describe(P.HYDRA_WS_FWD, cu, h, h_kv, d_qk, pairs, causal, tables=True)
    items = raw[plan["off_items2"]:][:plan["items2"] * ITEM.itemsize].view(ITEM)
    segs = raw[plan["off_segs"]:][:plan["segs"] * SEG.itemsize].view(SEG)
    return plan, items, segs


def rows_of(item, segs):
    """(to_part, output row) of each row of a tile, as the kernel finds them."""
    r = np.arange(int(item["rows"]))
    to_part, row = np.full(len(r), bool(item["to_part"])), int(item["out_row0"]) + r
    first, n = int(item["first_seg"]), int(item["n_segs"])
    assert first + n <= len(segs) or n == 0
    for s in segs[first:first + n]:
        at = r >= s["begin"]
        to_part[at], row[at] = bool(s["to_part"]), int(s["delta"]) + r[at]
    return to_part, row


@pytest.mark.parametrize("turned", [False, True])
@pytest.mark.parametrize("lengths,cp_r,h", [
    ([121] * 6, 2, 3), ([7, 300, 129, 16], 4, 2), ([290] * 40, 1, 6), ([1280], 1, 16), ([1280, 30], [2, 0], 20), ([700, 1, 64], 0, 4),
])
def test_every_row_goes_to_its_own_pair_once(all_pairs_short, lengths, cp_r, h, turned):
    cu = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    pairs, rows, _, _ = P.hydra_zigzag_pairs(cu, cp_r)
    if turned:                                         # groups may be listed in any order
        pairs = pairs[::-1].copy()
        pairs["group"] = pairs["group"].max() - pairs["group"]
    plan, items, segs = tables(cu, h, pairs)
    assert plan["items"] == 0
    seen = {True: np.zeros((h, rows), np.int64), False: np.zeros((h, int(cu[-1])), np.int64)}
    want = {True: np.zeros(rows, np.int64), False: np.zeros(int(cu[-1]), np.int64)}
    source = {True: np.zeros((rows, 3), np.int64), False: np.zeros((int(cu[-1]), 3), np.int64)}   # query, first key, keys
    for p in pairs:
        q0, n = int(cu[p["seq"]]) + int(p["q_start"]), int(p["q_len"])
        part = bool(p["part_row"] >= 0)
        at = int(p["part_row"]) if part else q0
        want[part][at:at + n] += 1
        source[part][at:at + n, 0] = q0 + np.arange(n)
        source[part][at:at + n, 1:] = int(cu[p["seq"]]) + int(p["k_start"]), int(p["k_len"])
    for it in items:
        if it["half"] == 2 or it["rows"] == 0:         # the other part of a tile whose first part is listed too
            continue
        for r, (part, row) in enumerate(zip(*rows_of(it, segs))):
            part = bool(part)
            seen[part][it["head"], row] += 1
            assert tuple(source[part][row]) == (int(it["q_tok0"]) + r, int(it["k_tok0"]), int(it["k_len"]))
    for part in (True, False):
        assert (seen[part] == want[part][None, :]).all()


def test_a_table_of_more_than_2_to_the_23_entries(all_pairs_short):
    """512 chunks of 2^21 - 1 rows that meet the same 64 keys: 2^23 shared tiles. The last ones' entries are their own."""
    n, size = 512, (1 << 21) - 1
    cu = np.array([0, n * size], dtype=np.int32)
    pairs = np.zeros(n, dtype=P.PAIR_DTYPE)
    pairs["q_start"] = pairs["part_row"] = np.arange(n) * size
    pairs["q_len"], pairs["k_len"], pairs["group"] = size, 64, np.arange(n)
    plan, items, segs = tables(cu, 1, pairs)
    assert plan["segs"] > 1 << 23
    assert (items["n_segs"] >= 1).all() and (items["first_seg"].astype(np.int64) + items["n_segs"] <= plan["segs"]).all()
    order = np.argsort(items["q_tok0"])
    for it in items[order[-600:]]:
        part, row = rows_of(it, segs)
        assert part.all() and (row == int(it["q_tok0"]) + np.arange(int(it["rows"]))).all()
