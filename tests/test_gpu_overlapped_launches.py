"""Launches of the library overlap at their ends with the launches around them on the same stream. What that must not touch:
kernels of others. Here torch writes the inputs right before each call and reads the results right behind it, call after
call without waiting for the GPU in between, and in a captured graph; every result must be bit-identical to the one of the
same calls made one at a time, with the GPU idle before each.
"""
import numpy as np
import pytest
import torch

import hydra_workloads as hw

pytestmark = pytest.mark.gpu
DQK, DV = hw.D_QK, hw.D_V


def normal(seed, *shape):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)


def new(*shape, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda")


class Attention:
    """Forward (and merge) and backward; with grouped K / V heads dk and dv are sums in no fixed order and are left out."""

    def __init__(self, lengths, h, cp_r=0, kv_heads=None, d_qk=DQK):
        import paper_2609_34318_b200 as P
        self.P, self.cu, self.h, self.kv, self.d = P, hw.cu_seqlens(lengths), h, kv_heads or h, d_qk
        T, self.pairs, self.rows = int(self.cu[-1]), None, 0
        if cp_r:
            self.pairs, self.rows, _, _ = P.hydra_zigzag_pairs(self.cu, cp_r)
        self.shapes = [(T, h, d_qk), (T, self.kv, d_qk), (T, self.kv, DV), (T, h, DV)]
        self.inputs = [new(*s) for s in self.shapes]
        self.out, self.lse, self.dq = new(T, h, DV), new(h, T, dtype=torch.float32), new(T, h, d_qk)
        self.dk, self.dv = new(T, self.kv, d_qk), new(T, self.kv, DV)
        self.o_part = new(self.rows, h, DV) if self.rows else None
        self.lse_part = new(h, self.rows, dtype=torch.float32) if self.rows else None
        ws = max(P.hydra_workspace_bytes_dims(w, self.cu, h, self.kv, d_qk, DV, self.pairs)
                 for w in (P.HYDRA_WS_FWD, P.HYDRA_WS_MERGE, P.HYDRA_WS_BWD))
        self.ws = torch.zeros(ws, dtype=torch.uint8, device="cuda")
        self.outputs = [self.out, self.lse, self.dq] + ([self.dk, self.dv] if self.kv == h else [])

    def calls(self):
        P, (q, k, v, do), scale = self.P, self.inputs, 1.0 / np.sqrt(self.d)
        dims = (self.cu, self.h, self.kv, self.d, DV, self.pairs, True, scale)
        yield lambda: P.hydra_attn_fwd_dims(q, k, v, *dims, self.out, self.lse, self.o_part, self.lse_part, self.rows, self.ws)
        if self.rows:
            yield lambda: P.hydra_lse_merge(self.o_part, self.lse_part, self.rows, self.cu, self.h, self.pairs, self.out,
                                            self.lse, self.ws)
        yield lambda: P.hydra_attn_bwd_dims(q, k, v, self.out, self.lse, do, *dims, self.dq, self.dk, self.dv, self.ws)


class Block:
    """The steps around the attention of an MLA block, each reading what the one before has written where it can."""

    def __init__(self, t, h, u, nope, rope, dv):
        import paper_2609_34318_b200 as P
        self.P, self.t, self.h, self.u, self.dims = P, t, h, u, (nope, rope, dv)
        self.shapes = [(t, h, nope + rope), (t, h, nope + dv), (t, rope), (t, h, dv)]
        self.inputs = [new(*s) for s in self.shapes]
        self.pos = torch.arange(t, dtype=torch.int32, device="cuda")
        self.q_rot, self.k, self.dq = (new(t, h, nope + rope) for _ in range(3))
        self.v, self.send, self.back, self.y, self.d_out, self.d_gate = (new(t, h, dv) for _ in range(6))
        self.dkv, self.dpe = new(t, h, nope + dv), new(t, rope)
        self.outputs = [self.q_rot, self.k, self.v, self.send, self.back, self.y, self.d_out, self.d_gate, self.dkv, self.dpe,
                        self.dq]

    def calls(self):
        P, t, h, u, (nope, rope, dv), (q, kv, pe, gate) = self.P, self.t, self.h, self.u, self.dims, self.inputs
        yield lambda: P.hydra_mla_rope(q, self.pos, t, h, nope + rope, nope, rope, 1e4, False, self.q_rot)
        yield lambda: P.hydra_mla_kv_assemble(kv, pe, self.pos, t, h, nope, rope, dv, 1e4, self.k, self.v)
        yield lambda: P.hydra_ulysses_pack(self.v, t, h, dv, u, self.send)
        yield lambda: P.hydra_ulysses_unpack(self.send, t, h, dv, u, self.back)
        yield lambda: P.hydra_gate_apply(self.back, gate, t * h * dv, self.y)
        yield lambda: P.hydra_gate_apply_bwd(self.y, self.back, gate, t * h * dv, self.d_out, self.d_gate)
        yield lambda: P.hydra_mla_kv_assemble_bwd(self.k, self.d_out, self.pos, t, h, nope, rope, dv, 1e4, self.dkv, self.dpe)
        yield lambda: P.hydra_mla_rope(self.q_rot, self.pos, t, h, nope + rope, nope, rope, 1e4, True, self.dq)


WORK = {
    "four short sequences": lambda: Attention([7, 33, 128, 300], 4),                     # halved tiles
    "a clustered backward": lambda: Attention([1300], 3),
    "both forward kernels": lambda: Attention([3000] + [300] * 60, 2),
    "cut and merged": lambda: Attention([300, 700, 64], 6, cp_r=1),
    "grouped heads of 128": lambda: Attention([900, 200, 77], 8, kv_heads=2, d_qk=128),
    "MLA block": lambda: Block(700, 24, 4, 128, 64, 128),
    "MLA block, odd dimensions": lambda: Block(700, 24, 4, 126, 62, 120),
}


def one_pass(work, src, wait=lambda: None):
    """The inputs are written, the outputs poisoned, the calls made and the results copied, all on the current stream."""
    for dst, x in zip(work.inputs, src):
        dst.copy_(x)
    for o in work.outputs:
        o.fill_(float("nan"))
    for call in work.calls():
        wait()
        call()
        wait()
    return [o.clone() for o in work.outputs]


def same(a, b):
    return all(torch.equal(x.view(torch.uint8), y.view(torch.uint8)) for x, y in zip(a, b))


@pytest.mark.parametrize("name", list(WORK))
def test_others_kernels_right_before_and_behind(name):
    work = WORK[name]()
    sources = [[normal(100 * s + i, *shape) for i, shape in enumerate(work.shapes)] for s in range(3)]
    alone = [one_pass(work, src, torch.cuda.synchronize) for src in sources]
    torch.cuda.synchronize()
    got = [one_pass(work, sources[i % 3]) for i in range(24)]
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert same(g, alone[i % 3]), (name, i)


@pytest.fixture
def no_tables():
    """Work tables reach the device on the stream that asks first, and a capture cannot wait for another stream."""
    import paper_2609_34318_b200 as P
    torch.cuda.synchronize()
    P.hydra_shutdown()
    yield
    torch.cuda.synchronize()
    P.hydra_shutdown()


@pytest.mark.parametrize("name", list(WORK))
def test_in_a_captured_graph(name, no_tables):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        work = WORK[name]()
        sources = [[normal(100 * s + i, *shape) for i, shape in enumerate(work.shapes)] for s in range(2)]
        alone = [one_pass(work, src, torch.cuda.synchronize) for src in sources]
        held = [x.clone() for x in sources[0]]
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            results = one_pass(work, held)
        for i in range(8):
            for dst, x in zip(held, sources[i % 2]):
                dst.copy_(x)
            graph.replay()
            graph.replay()
            got = [r.clone() for r in results]
            stream.synchronize()
            assert same(got, alone[i % 2]), (name, i)
