"""The backward over pairs that stay as they are listed, because something of a sequence's causal triangle is missing, there is
no mask, or the tensors are local: work items that visit several pairs, of one query head and of several, one-shot, in bands and
accumulating, with dS handed over and recomputed. Against the oracle's sums over the same pairs."""
import functools

import numpy as np
import pytest
import torch

import hydra_workloads as hw
import oracle
from gpu_util import check

pytestmark = pytest.mark.gpu
DV = hw.D_V


def listed(cu, cp_r, causal, left_out):
    """Chunk pairs of every sequence: those that the mask shows, or all of them, without the left_out-th of each sequence."""
    import paper_2609_34318_b200 as P
    pairs, _, _, _ = P.hydra_zigzag_pairs(cu, cp_r)
    out = []
    for b in range(len(cu) - 1):
        chunks = sorted({(int(p["q_start"]), int(p["q_len"])) for p in pairs if p["seq"] == b})
        own = [(b, *q, *k) for q in chunks for k in chunks if not causal or k[0] <= q[0]]
        out += [p for i, p in enumerate(own) if i != left_out]
    return np.array([(*p, -1, i, 0) for i, p in enumerate(out)], dtype=P.PAIR_DTYPE)


@functools.lru_cache(maxsize=None)
def problem(lengths, h, h_kv, d_qk, cp_r, causal, left_out):
    """Inputs, pairs, out and lse of the whole problem and the gradients of the listed pairs (the forms share them)."""
    cu = hw.cu_seqlens(list(lengths))
    rng = np.random.default_rng(len(lengths) + h)
    f = lambda heads, d: hw.f32_to_bf16_bits(rng.standard_normal((int(cu[-1]), heads, d)).astype(np.float32))
    x = dict(q=f(h, d_qk), k=f(h_kv, d_qk), v=f(h_kv, DV), do=f(h, DV))
    scale = np.float32(1.0 / np.sqrt(np.float32(d_qk)))
    pairs = listed(cu, list(cp_r) if isinstance(cp_r, tuple) else cp_r, causal, left_out)
    out, lse = oracle.attn_fwd_gqa(x["q"], x["k"], x["v"], cu, causal, scale)
    out = torch.from_numpy(out.astype(np.float32)).to(torch.bfloat16)
    ora = [{n: int(p[n]) for n in ("seq", "q_start", "q_len", "k_start", "k_len")} for p in pairs]
    ref = oracle.attn_bwd_pairs_gqa(x["q"], x["k"], x["v"], x["do"], cu, ora, causal, scale, lse,
                                    oracle.bwd_prep(x["do"], out.double().numpy()))
    return cu, x, scale, pairs, out, torch.from_numpy(lse.astype(np.float32)), dict(zip(("dq", "dk", "dv"), ref))


@pytest.fixture(params=["hand_off", "recompute", "bands"])
def form(request):
    import paper_2609_34318_b200 as P
    P.hydra_set_bwd_scratch_limit({"hand_off": 4 << 30, "recompute": 0, "bands": 1 << 20}[request.param])
    P.hydra_set_bwd_band_scratch(1 << 20 if request.param == "bands" else 0)
    yield request.param
    P.hydra_set_bwd_scratch_limit(4 << 30)
    P.hydra_set_bwd_band_scratch(P.HYDRA_BAND_AUTO)


CASES = [
    # lengths, heads, K / V heads, d_qk, ring, causal, left out, query heads per key-side item
    ((300,) * 24, 8, 2, 192, 2, True, 3, 4),       # a whole group per item, up to four pairs
    ((200,) * 30, 8, 2, 128, 2, True, 3, 4),
    ((290,) * 24, 8, 1, 192, 1, False, None, 8),
    ((600,) * 6, 16, 1, 128, 2, True, 3, 4),       # four items add into the rows of a K / V head
    ((512,) * 8, 16, 1, 192, 1, False, None, 4),
    ((300,) * 14, 4, 4, 192, 2, True, 3, 1),       # a K / V head per query head, ragged chunks of 75 rows
    ((1500, 640), 2, 2, 192, (2, 1), True, 1, 1),  # few tiles: two CTAs share one
    ((900, 333), 2, 2, 192, (1, 2), False, None, 1),
    ((900, 333), 3, 3, 128, (1, 2), False, 3, 1),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{len(c[0])}x{c[0][0]}-{c[1]}/{c[2]}-{c[3]}-{c[5]}-{c[6]}")
def test_listed_pairs(case, form):
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import bits_to_tensor
    *args, item_heads = case
    lengths, h, h_kv, d_qk, _, causal, _ = args
    if form == "bands" and h != h_kv:
        pytest.skip("bands are for a K / V head per query head")
    cu, x, scale, pairs, out, lse, ref = problem(*args)
    plan = P.hydra_plan_describe(P.HYDRA_WS_BWD, cu, h, h_kv, d_qk, pairs, causal)
    assert plan["pairs"] == len(pairs) and plan["item_heads"] == item_heads
    q, k, v, do = (bits_to_tensor(x[n]) for n in ("q", "k", "v", "do"))
    need = P.hydra_workspace_bytes_dims(P.HYDRA_WS_BWD, cu, h, h_kv, d_qk, DV, pairs)
    # (sized for a causal call; without a mask a form takes more)
    if form == "hand_off":
        need += sum(2 * int(p["q_len"] + 192) * int(p["k_len"] + 192) for p in pairs) * h
    elif form == "bands":
        need += 4 * d_qk * int(cu[-1]) * h + (2 << 20)
    ws = torch.randint(0, 255, (need,), dtype=torch.uint8, device="cuda")
    g = [torch.full((int(cu[-1]), heads, d), float("nan"), dtype=torch.bfloat16, device="cuda")
         for heads, d in ((h, d_qk), (h_kv, d_qk), (h_kv, DV))]
    n0 = P.hydra_launch_count()
    P.hydra_attn_bwd_dims(q, k, v, out.cuda(), lse.cuda(), do, cu, h, h_kv, d_qk, DV, pairs, causal, float(scale), *g, ws)
    launches = P.hydra_launch_count() - n0
    status, detail = P.hydra_poll_status(ws)
    assert status == 0, (status, detail)
    if form == "bands":
        n_bands = P.hydra_bwd_bands(cu, h, pairs, causal, 1 << 20)[2]
        assert n_bands >= 2 and launches >= 1 + 2 * n_bands + 1
    got = {n: t.float().cpu().numpy().astype(np.float64) for n, t in zip(("dq", "dk", "dv"), g)}
    check(got, ref, names=("dq", "dk", "dv"), label=f"{case} {form}: ")


@pytest.mark.parametrize("case", [CASES[0], CASES[3], CASES[6]], ids=["whole group", "part of a group", "per head"])
@pytest.mark.parametrize("recompute", [False, True])
def test_listed_pairs_of_local_tensors(case, recompute):
    """The accumulating form on tensors that hold the chunks in an order of their own; twice into the same sums."""
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import bits_to_tensor
    *args, _ = case
    lengths, h, h_kv, d_qk, _, causal, _ = args
    cu, x, scale, pairs, out, lse, ref = problem(*args)
    T = int(cu[-1])
    def table(seed):
        """Chunks in another order, three rows apart, and the tensor row of every token."""
        chunks = sorted({(int(p["seq"]), int(p["q_start"]), int(p["q_len"])) for p in pairs})
        rows, rng, at, tab = np.zeros(T, np.int64), np.random.default_rng(seed), 0, []
        for i in rng.permutation(len(chunks)):
            b, s, n = chunks[i]
            tab.append((b, s, n, at))
            rows[int(cu[b]) + s:int(cu[b]) + s + n] = at + np.arange(n)
            at += n + 3
        return tab, at, torch.from_numpy(rows).cuda()
    (qt, q_rows, qr), (kt, kv_rows, kr) = table(1), table(2)

    def local(t, n, r):
        into = torch.zeros((n,) + tuple(t.shape[1:]), dtype=t.dtype, device="cuda")
        into[r] = t.cuda()
        return into
    q, do, o = (local(t, q_rows, qr) for t in (bits_to_tensor(x["q"]), bits_to_tensor(x["do"]), out))
    k, v = (local(bits_to_tensor(x[n]), kv_rows, kr) for n in ("k", "v"))
    l = torch.zeros((h, q_rows), dtype=torch.float32, device="cuda")
    l[:, qr] = lse.cuda()
    P.hydra_set_bwd_scratch_limit(0 if recompute else 4 << 30)
    try:
        ws = torch.empty(P.hydra_workspace_bytes_local(P.HYDRA_WS_BWD, cu, h, h_kv, d_qk, DV, qt, q_rows, kt, kv_rows, pairs),
                         dtype=torch.uint8, device="cuda")
        acc = [torch.zeros((n, heads, d), dtype=torch.float32, device="cuda")
               for n, heads, d in ((q_rows, h, d_qk), (kv_rows, h_kv, d_qk), (kv_rows, h_kv, DV))]
        for _ in range(2):
            P.hydra_attn_bwd_accumulate_local(q, k, v, o, l, do, cu, h, h_kv, d_qk, DV, qt, q_rows, kt, kv_rows, pairs, causal,
                                              float(scale), *acc, ws)
        assert P.hydra_poll_status(ws)[0] == 0
    finally:
        P.hydra_set_bwd_scratch_limit(4 << 30)
    got = {n: (t[r] / 2).cpu().numpy().astype(np.float64) for n, t, r in zip(("dq", "dk", "dv"), acc, (qr, kr, kr))}
    check(got, ref, names=("dq", "dk", "dv"), label=f"local {case}: ")
