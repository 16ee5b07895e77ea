"""Forward calls with no more work items than slots, which run without the launch that clears the status block: whatever the
workspace held, results and status are those of a call in a clean one, on both sides of the line, also when replayed."""
import numpy as np
import pytest
import torch

import hydra_workloads as hw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,h", [([1], 1), ([7, 33, 128, 300], 4), ([128] * 37, 4), ([128] * 149, 1), ([100] * 74, 4),
                                       ([100] * 297, 1), ([900], 8)])
@pytest.mark.parametrize("fill", [0x00, 0xFF, 0x5A, None])
def test_any_workspace_will_do(lengths, h, fill):
    import paper_2609_34318_b200 as P
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(len(lengths))
    q, k, v = (torch.randn((T, h, d), generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)
               for d in (hw.D_QK, hw.D_QK, hw.D_V))
    scale = float(np.float32(1.0 / np.sqrt(np.float32(hw.D_QK))))

    def forward(ws, out, lse):
        P.hydra_attn_fwd(q, k, v, cu, h, None, True, scale, out, lse, None, None, 0, ws)

    def outputs():
        return (torch.full((T, h, hw.D_V), float("nan"), dtype=torch.bfloat16, device="cuda"),
                torch.full((h, T), float("nan"), dtype=torch.float32, device="cuda"))
    ref = outputs()
    clean = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    forward(clean, *ref)
    assert P.hydra_poll_status(clean)[0] == P.HYDRA_OK
    if fill is None:
        ws = torch.randint(0, 256, (4096,), dtype=torch.uint8, device="cuda")
    else:
        ws = torch.full((4096,), fill, dtype=torch.uint8, device="cuda")
    for _ in range(3):
        got = outputs()
        forward(ws, *got)
        assert P.hydra_poll_status(ws)[0] == P.HYDRA_OK
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    torch.cuda.synchronize()
    P.hydra_shutdown()                                 # (tables reach the device on the stream that asks first)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        got = outputs()
        forward(ws, *got)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            forward(ws, *got)
        for _ in range(2):
            got[0].fill_(float("nan"))
            got[1].fill_(float("nan"))
            graph.replay()
            stream.synchronize()
            assert P.hydra_poll_status(ws)[0] == P.HYDRA_OK
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    P.hydra_shutdown()


SMALL_NUMBERS = """
import numpy as np, torch
import hydra_workloads as hw
import paper_2609_34318_b200 as P
cu = hw.cu_seqlens([7, 33])
q, k, v = (torch.ones((40, 2, d), dtype=torch.bfloat16, device="cuda") for d in (hw.D_QK, hw.D_QK, hw.D_V))
out, lse = torch.empty((40, 2, hw.D_V), dtype=torch.bfloat16, device="cuda"), torch.empty((2, 40), device="cuda")
got = []
for n in range(1, 9):                                  # the workspace held int32 tensors (positions, token ids) before
    ws = torch.full((1024,), n, dtype=torch.int32, device="cuda").view(torch.uint8)
    P.hydra_attn_fwd(q, k, v, cu, 2, None, True, 0.07, out, lse, None, None, 0, ws)
    got.append(P.hydra_poll_status(ws)[0])
print(got)
assert got == [P.HYDRA_OK] * 8
"""


def test_small_numbers_in_the_workspace_are_no_error():
    """The first calls of a process, in workspaces that hold a small number all over: the number of the call must not be one
    that ordinary data hold."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", SMALL_NUMBERS], capture_output=True, text=True, timeout=300, cwd=root)
    assert run.returncode == 0, run.stdout + run.stderr
