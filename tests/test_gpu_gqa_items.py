"""Key-side items that take several query heads of a K / V head (calls with many key tiles) and the sums in fp32 that other
calls need, against the oracle: whole groups, part of a group, ragged tiles, cut sequences (whose pairs are joined; several pairs
per item: test_gpu_listed_pairs_backward), heads of 192 and of 128."""
import numpy as np
import pytest

import hydra_workloads as hw
import oracle
from gpu_util import check, pairs_for

pytestmark = pytest.mark.gpu
DV = hw.D_V


@pytest.mark.parametrize("lengths,h,h_kv,d_qk,cp_r,item_heads", [
    ([130] * 50, 8, 2, 192, 0, 4),                 # 100 tiles of 2 K / V heads: every item holds a whole group
    ([257, 64, 300] * 14, 8, 1, 128, 0, 4),        # two items per group
    ([300] * 24, 4, 2, 192, 1, 2),                 # cut sequences, whose pairs are joined
    ([1500, 700], 8, 2, 192, 0, 1),                # few long tiles: an item per query head, summed in fp32
    ([600] * 8, 16, 1, 128, 0, 4),                 # four items per group, summed in fp32
    ([129, 1, 64], 4, 1, 128, 0, 4),               # fewer tiles than SMs
])
def test_items_of_several_query_heads(lengths, h, h_kv, d_qk, cp_r, item_heads):
    import torch
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import bits_to_tensor
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    rng = np.random.default_rng(len(lengths) * 100 + h)
    x = {n: hw.f32_to_bf16_bits(rng.standard_normal((T, heads, d)).astype(np.float32))
         for n, heads, d in (("q", h, d_qk), ("k", h_kv, d_qk), ("v", h_kv, DV), ("do", h, DV))}
    lib_pairs, rows, ora_pairs = pairs_for(cu, cp_r) if cp_r else (None, 0, None)
    assert P.hydra_plan_describe(P.HYDRA_WS_BWD, cu, h, h_kv, d_qk, lib_pairs)["item_heads"] == item_heads
    scale = float(np.float32(1.0 / np.sqrt(np.float32(d_qk))))
    q, k, v, do = (bits_to_tensor(x[n]) for n in ("q", "k", "v", "do"))
    out = torch.empty((T, h, DV), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((h, T), dtype=torch.float32, device="cuda")
    o_part = torch.empty((max(rows, 1), h, DV), dtype=torch.bfloat16, device="cuda")
    lse_part = torch.empty((h, max(rows, 1)), dtype=torch.float32, device="cuda")
    need = max(P.hydra_workspace_bytes_dims(w, cu, h, h_kv, d_qk, DV, lib_pairs)
               for w in (P.HYDRA_WS_FWD, P.HYDRA_WS_MERGE, P.HYDRA_WS_BWD))
    ws = torch.randint(0, 255, (need,), dtype=torch.uint8, device="cuda")      # what is added into has to be cleared
    P.hydra_attn_fwd_dims(q, k, v, cu, h, h_kv, d_qk, DV, lib_pairs, True, scale, out, lse, o_part if rows else None,
                          lse_part if rows else None, rows, ws)
    if rows:
        P.hydra_lse_merge(o_part, lse_part, rows, cu, h, lib_pairs, out, lse, ws)
    got = []
    for _ in range(2):
        g = [torch.full((T, heads, d), float("nan"), dtype=torch.bfloat16, device="cuda")
             for heads, d in ((h, d_qk), (h_kv, d_qk), (h_kv, DV))]
        P.hydra_attn_bwd_dims(q, k, v, out, lse, do, cu, h, h_kv, d_qk, DV, lib_pairs, True, scale, *g, ws)
        status, detail = P.hydra_poll_status(ws)
        assert status == 0, (status, detail)
        got.append(g)
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    o_ref, l_ref = oracle.attn_fwd_gqa(x["q"], x["k"], x["v"], cu, True, np.float32(scale))
    if ora_pairs is None:
        ref = oracle.attn_bwd_gqa(x["q"], x["k"], x["v"], x["do"], cu, True, np.float32(scale), o_ref, l_ref)
    else:
        ref = oracle.attn_bwd_pairs_gqa(x["q"], x["k"], x["v"], x["do"], cu, ora_pairs, True, np.float32(scale), l_ref,
                                        oracle.bwd_prep(x["do"], o_ref))
    for g in got:
        check(dict(out=f64(out), lse=f64(lse), dq=f64(g[0]), dk=f64(g[1]), dv=f64(g[2])),
              dict(out=o_ref, lse=l_ref, dq=ref[0], dk=ref[1], dv=ref[2]), label=f"{len(lengths)} sequences, {h}/{h_kv} heads: ")
    # one item per row: nothing is added in memory; two: both orders of two additions to zero give the same sum
    if h // h_kv <= 2 * item_heads:
        for a, b in zip(*got):
            assert torch.equal(a, b)
