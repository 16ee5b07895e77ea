"""The merge with several thread blocks per eight rows of a chunk (calls of few rows), against the oracle."""
import numpy as np
import pytest
import torch

import hydra_workloads as hw
from gpu_util import oracle_merge_of_partials
from test_gpu_merge import _compare, _fill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,cp_r,h", [([40, 9, 1], 1, 64), ([130], 2, 33), ([600], 4, 16), ([2400], 1, 32), ([8], 1, 5)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_merge_shared_by_thread_blocks(lengths, cp_r, h, accumulate):
    import paper_2609_34318_b200 as P
    rng = np.random.default_rng(h)
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    pairs, part_rows, _, _ = P.hydra_zigzag_pairs(cu, cp_r)
    o_part, lse_part, _ = _fill(rng, part_rows, h, 0.2, 4.0)
    out0, lse0, _ = _fill(rng, T, h, 0.2, 4.0)
    out, lse = out0.clone(), lse0.clone()
    ws = torch.empty(4096, dtype=torch.uint8, device="cuda")
    merge = P.hydra_lse_merge_accumulate if accumulate else P.hydra_lse_merge
    merge(o_part, lse_part, part_rows, cu, h, pairs, out, lse, ws)
    torch.cuda.synchronize()
    current = dict(out_cur=out0.float().cpu().numpy().astype(np.float64),
                   lse_cur=lse0.cpu().numpy().astype(np.float64)) if accumulate else {}
    ref_out, ref_lse = oracle_merge_of_partials(cu, pairs, o_part, lse_part, T, h, **current)
    _compare(out, lse, ref_out, ref_lse, f"{lengths} {cp_r} {h}")
