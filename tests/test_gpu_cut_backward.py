"""The backward of cut sequences: pairs that cover whole sequences run as the uncut problem, others pair by pair."""
import numpy as np
import pytest
import torch

import hydra_workloads as hw
from gpu_util import check, pairs_for, run_gpu, run_oracle

pytestmark = pytest.mark.gpu
DV = hw.D_V


def tensors(cu, h, seed):
    rng = np.random.default_rng(seed)
    f = lambda d: hw.f32_to_bf16_bits(rng.standard_normal((int(cu[-1]), h, d)).astype(np.float32))
    return dict(q=f(hw.D_QK), k=f(hw.D_QK), v=f(DV), do=f(DV))


@pytest.mark.parametrize("lengths,cp_r,left_out", [
    ([300, 129, 64], [1, 2, 0], []),               # all whole
    ([700], [2], [5]),                             # one pair missing: pair by pair
    ([640, 200, 333], [4, 1, 2], [3, 20]),         # one sequence whole, pairs of others missing
])
def test_cut_backward_matches_the_oracle(lengths, cp_r, left_out):
    cu, h = hw.cu_seqlens(lengths), 2
    x = tensors(cu, h, 5 + len(lengths))
    pairs, rows, ora = pairs_for(cu, cp_r)
    got = run_gpu(x, cu, h, pairs, rows)
    check(got, run_oracle(x, cu, pairs=ora), label=f"{lengths} {cp_r}: ")
    if not left_out:
        return
    import oracle
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import bits_to_tensor
    keep = [i for i in range(len(pairs)) if i not in left_out]
    some, ora_some = pairs[keep].copy(), [ora[i] for i in keep]
    scale = float(np.float32(1.0 / np.sqrt(np.float32(hw.D_QK))))
    q, k, v, do = (bits_to_tensor(x[n]) for n in ("q", "k", "v", "do"))
    ref = run_oracle(x, cu, pairs=ora)                 # (out and lse of the whole problem, gradients of some of its pairs)
    out = torch.from_numpy(ref["out"].astype(np.float32)).to(torch.bfloat16).cuda()
    lse = torch.from_numpy(ref["lse"].astype(np.float32)).cuda()
    ws = torch.empty(P.hydra_workspace_bytes(P.HYDRA_WS_BWD, cu, h, some), dtype=torch.uint8, device="cuda")
    grads = [torch.zeros(tuple(q.shape[:2]) + (d,), dtype=torch.bfloat16, device="cuda") for d in (hw.D_QK, hw.D_QK, DV)]
    P.hydra_attn_bwd(q, k, v, out, lse, do, cu, h, some, True, scale, *grads, ws)
    assert P.hydra_poll_status(ws)[0] == 0
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    out_r = f64(out)
    dq, dk, dv = oracle.attn_bwd_pairs(x["q"], x["k"], x["v"], x["do"], cu, ora_some, True, np.float32(scale), ref["lse"],
                                       oracle.bwd_prep(x["do"], out_r))
    check(dict(dq=f64(grads[0]), dk=f64(grads[1]), dv=f64(grads[2])), dict(dq=dq, dk=dk, dv=dv), names=("dq", "dk", "dv"),
          label=f"{lengths} without {left_out}: ")
