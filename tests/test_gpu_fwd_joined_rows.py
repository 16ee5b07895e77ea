"""Forward of sequences cut into chunks shorter than a tile: consecutive q chunks share the tiles of a kv chunk and every row goes
to its own pair's output. Each pair's partial against the oracle's for that pair, and the merged result."""
import numpy as np
import pytest
import torch

import hydra_workloads as hw
import oracle
from gpu_util import TOL_LSE, TOL_REL, check, pairs_for, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,h,cp_r,causal", [
    ([121] * 3, 4, 2, True),                       # four chunks of 30 rows in one tile
    ([121] * 40, 8, 2, True),                      # more tiles than SMs
    ([7, 300, 129, 16], 3, 4, True),               # chunks of no row, of one, of 37
    ([290] * 30, 6, 1, True),                      # a chunk's 17 rows beyond its first tile ride with the next chunk's
    ([500, 260], 2, 2, False),
    ([128, 256], 2, 1, True),                      # 64 and 128 rows: one tile is saved, none
])
def test_rows_of_several_pairs_in_a_tile(lengths, h, cp_r, causal):
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import bits_to_tensor
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    rng = np.random.default_rng(T)
    f = lambda d: hw.f32_to_bf16_bits(rng.standard_normal((T, h, d)).astype(np.float32))
    x = dict(q=f(hw.D_QK), k=f(hw.D_QK), v=f(hw.D_V), do=f(hw.D_V))
    pairs, rows, ora = pairs_for(cu, cp_r)
    scale = float(np.float32(1.0 / np.sqrt(np.float32(hw.D_QK))))
    q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
    nan = float("nan")
    out = torch.full((T, h, hw.D_V), nan, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((h, T), nan, dtype=torch.float32, device="cuda")
    o_part = torch.full((rows + 64, h, hw.D_V), nan, dtype=torch.bfloat16, device="cuda")
    lse_part = torch.full((h, rows + 64), nan, dtype=torch.float32, device="cuda")
    ws = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    P.hydra_attn_fwd(q, k, v, cu, h, pairs, causal, scale, out, lse, o_part, lse_part, rows + 64, ws)
    assert P.hydra_poll_status(ws)[0] == P.HYDRA_OK
    assert torch.isnan(lse_part[:, rows:]).all() and torch.isnan(o_part[rows:].float()).all()
    # every pair by itself: its rows against its keys
    qf, kf, vf = (bits_to_tensor(x[n]).double().cpu().numpy() for n in ("q", "k", "v"))
    o_np, l_np = o_part.double().cpu().numpy(), lse_part.double().cpu().numpy()
    out_np, lse_np = out.double().cpu().numpy(), lse.double().cpu().numpy()
    for p in pairs:
        n = int(p["q_len"])
        if n == 0:
            continue
        t0, k0 = int(cu[p["seq"]]) + int(p["q_start"]), int(cu[p["seq"]]) + int(p["k_start"])
        s = np.einsum("qhd,khd->hqk", qf[t0:t0 + n], kf[k0:k0 + int(p["k_len"])]) * scale
        if causal:
            s[:, np.arange(int(p["q_start"]), int(p["q_start"]) + n)[:, None] < np.arange(int(p["k_start"]), int(p["k_start"]) + int(p["k_len"]))] = -np.inf
        m = s.max(-1, keepdims=True)
        e = np.exp(s - m)
        ref_l = (m + np.log(e.sum(-1, keepdims=True)))[..., 0]
        ref_o = np.einsum("hqk,khd->qhd", e / e.sum(-1, keepdims=True), vf[k0:k0 + int(p["k_len"])])
        pr = int(p["part_row"])
        got_o, got_l = (o_np[pr:pr + n], l_np[:, pr:pr + n]) if pr >= 0 else (out_np[t0:t0 + n], lse_np[:, t0:t0 + n])
        assert np.abs(got_l - ref_l).max() <= TOL_LSE, p
        assert np.abs(got_o - ref_o).max() <= TOL_REL * max(1.0, np.abs(ref_o).max()), p
    if causal:
        P.hydra_lse_merge(o_part, lse_part, rows + 64, cu, h, pairs, out, lse, ws)
        got = dict(out=out.double().cpu().numpy(), lse=lse.double().cpu().numpy())
        check(got, run_oracle(x, cu, pairs=ora, backward=False), names=("out", "lse"), label=f"{lengths[:3]} {cp_r}: ")
