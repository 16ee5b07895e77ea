"""Forward calls of a few q tiles per SM, whose thread blocks run several tiles with the keys of the longer ones shared by both
slots, against the oracle; twice, bit for bit (a tile's second part stands in shared memory that the next tile is loaded into)."""
import numpy as np
import pytest
import torch

import hydra_workloads as hw
import oracle
from gpu_util import check, pairs_for
from test_plan_tables import tables

pytestmark = pytest.mark.gpu


# shared: the most shared tiles of a thread block on 148 SMs, 0: the call goes to the queue
@pytest.mark.parametrize("lengths,h,h_kv,d_qk,cp_r,causal,shared", [
    ([1300], 16, 16, 192, 0, True, 1),             # 176 tiles, the longest in 21 steps
    ([1100, 383, 64, 7, 129], 12, 12, 192, 0, True, 1),    # long and short tiles in one call
    ([1537], 18, 2, 128, 0, True, 2),
    ([2050], 14, 14, 192, 0, True, 2),             # the last tile has two rows
    ([1280], 20, 4, 192, 1, True, 0),              # chunk pairs, merged
    ([900, 500], 14, 14, 128, 0, False, 2),
    ([10240], 4, 2, 128, 0, True, 3),              # the waits on a part come round to their first phase again
    ([7992], 1, 1, 128, 2, True, 2),               # cut: tiles that hold rows of several pairs, shared
    ([8166, 2216], 1, 1, 192, 2, True, 3),
    ([3391, 7186], 2, 2, 192, [2, 1], True, 4),
])
def test_tiles_dealt_out_and_shared(lengths, h, h_kv, d_qk, cp_r, causal, shared):
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import bits_to_tensor
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    rng = np.random.default_rng(T)
    x = {n: hw.f32_to_bf16_bits(rng.standard_normal((T, heads, d)).astype(np.float32))
         for n, heads, d in (("q", h, d_qk), ("k", h_kv, d_qk), ("v", h_kv, hw.D_V))}
    pairs, rows, _ = pairs_for(cu, cp_r) if cp_r else (None, 0, None)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        plan, items, segs = tables(cu, h, pairs, causal, h_kv, d_qk)
        halves = items.reshape(-1, 2, plan["grid"])[:, 0]["half"] if plan["shared"] else np.zeros((1, 1))
        assert (halves == 1).sum(axis=0).max() == shared
        assert (len(segs) > 0) == (cp_r != 0 and shared > 0)
    scale = float(np.float32(1.0 / np.sqrt(np.float32(d_qk))))
    q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
    ws = torch.randint(0, 256, (4096,), dtype=torch.uint8, device="cuda")
    got = []
    for _ in range(2):
        out = torch.full((T, h, hw.D_V), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((h, T), float("nan"), dtype=torch.float32, device="cuda")
        o_part = torch.full((max(rows, 1), h, hw.D_V), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse_part = torch.full((h, max(rows, 1)), float("nan"), dtype=torch.float32, device="cuda")
        P.hydra_attn_fwd_dims(q, k, v, cu, h, h_kv, d_qk, hw.D_V, pairs, causal, scale, out, lse, o_part if rows else None,
                              lse_part if rows else None, rows, ws)
        assert P.hydra_poll_status(ws)[0] == P.HYDRA_OK
        if rows:
            P.hydra_lse_merge(o_part, lse_part, rows, cu, h, pairs, out, lse, ws)
        got.append((out, lse))
    ref_out, ref_lse = oracle.attn_fwd_gqa(x["q"], x["k"], x["v"], cu, causal, np.float32(scale))
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    check(dict(out=f64(got[0][0]), lse=f64(got[0][1])), dict(out=ref_out, lse=ref_lse), names=("out", "lse"),
          label=f"{lengths} {h}/{h_kv} heads of {d_qk}: ")
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
