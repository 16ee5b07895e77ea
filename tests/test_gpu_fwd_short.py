"""The short-sequence forward kernel and the routing between the two forward kernels.

Section 2.2 of the paper: most sequences of a training batch are short. Pairs whose q and kv ranges are at most
`hydra_set_fwd_short_len` tokens long go to a kernel of their own (one CTA per SM, two independent 128-row q
tiles in flight, steps of 64 keys); the others stay on the CTA-pair kernel; a call whose short pairs carry less
than a quarter of its work uses the CTA-pair kernel alone. Every case here is checked against the fp64 oracle
(the small parity cases of the other test files run on both kernels as well: fixture `both_forward_kernels`).
"""
import numpy as np
import pytest
import torch

import hydra_workloads as hw
from conftest import FWD_SHORT_LEN_DEFAULT
from gpu_util import TOL_LSE, TOL_REL, check, pairs_for, run_gpu, run_oracle

pytestmark = pytest.mark.gpu
DQK, DV = hw.D_QK, hw.D_V


def rand_inputs(seed, T, h):
    rng = np.random.default_rng(seed)
    f = lambda d: hw.f32_to_bf16_bits(rng.standard_normal((T, h, d)).astype(np.float32))
    return dict(q=f(DQK), k=f(DQK), v=f(DV), do=f(DV))


def forward_launches(fn):
    """Launches of the library's kernels made by fn()."""
    import paper_2609_34318_b200 as P
    before = P.hydra_launch_count()
    fn()
    return P.hydra_launch_count() - before


@pytest.fixture(autouse=True)
def default_routing():
    import paper_2609_34318_b200 as P
    P.hydra_set_fwd_short_len(FWD_SHORT_LEN_DEFAULT)
    yield
    P.hydra_set_fwd_short_len(FWD_SHORT_LEN_DEFAULT)


@pytest.mark.parametrize("lengths", [
    [7, 33, 128, 300],            # a tile with 7 rows, one of exactly 128, one sequence of three tiles
    [1, 1, 1, 2],                 # work items of a single row and a single key
    [63, 65, 64],                 # one key more and one key less than a step
    [129, 257, 64, 500, 127],     # one row more than a tile, one more than two
    [2048],                       # 16 tiles of up to 32 steps in halves
    [200] * 40,                   # more work items than the two slots of every SM hold at once
    [1024] * 7,                   # tiles of up to 16 steps, the longest call whose slots pop two items ahead throughout
    [1025] * 6,                   # one step more: popped near the end of an item (162 tiles: not a halved call either)
])
def test_short_sequences_against_the_oracle(lengths):
    h = 3
    cu = hw.cu_seqlens(lengths)
    x = rand_inputs(sum(lengths), int(cu[-1]), h)
    got = run_gpu(x, cu, h)
    ref = run_oracle(x, cu)
    check(got, ref, label=f"{lengths[:5]} ")


@pytest.mark.parametrize("lengths,h", [
    ([1], 1),                     # one row, one step: nothing for the second slot
    ([64], 2), ([65], 2),         # one step and two
    ([128], 3), ([129, 192], 2),  # two steps; three and four, rows that see nothing of the second part
    ([700, 33, 1], 3),            # an odd number of steps beside single ones
    ([3000], 2),                  # longer than the limit of the short-sequence kernel: 24 tiles, up to 47 steps
    ([128] * 37, 4),              # 148 tiles: as many as the GPU has SMs
    ([128] * 37 + [1], 4),        # one more: no halves
])
def test_tiles_shared_by_the_two_slots(lengths, h):
    """A call with no more q tiles than SMs gives each slot of a thread block half of a tile's keys. The two parts are
    joined in fp32 before the one rounding to bf16, so the tolerance is that of the whole tile."""
    cu = hw.cu_seqlens(lengths)
    x = rand_inputs(sum(lengths) + h, int(cu[-1]), h)
    got = run_gpu(x, cu, h)
    check(got, run_oracle(x, cu), label=f"{lengths[:4]} ")


@pytest.mark.parametrize("keys", [
    131070 * 64,              # the most that two halves of a tile count in 16 bits each (8.4M keys)
    131071 * 64 + 5,          # one step and a ragged one more: not a matter of this kernel any more
])
def test_as_many_keys_as_a_work_item_counts_and_more(keys):
    """A few q rows against millions of keys is a call with no more q tiles than SMs, which shares a tile's keys between
    two slots, as long as their steps of 64 keys fit the 16 bits of a work item."""
    import paper_2609_34318_b200 as P
    q_len = 3
    cu = np.array([0, keys], dtype=np.int32)
    gen = torch.Generator(device="cuda").manual_seed(keys)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    q, k, v = normal(q_len, 1, DQK), normal(keys, 1, DQK), normal(keys, 1, DV)
    pairs = [dict(seq=0, q_start=keys - q_len, q_len=q_len, k_start=0, k_len=keys, part_row=-1, group=0)]
    q_chunks, kv_chunks = [(0, keys - q_len, q_len, 0)], [(0, 0, keys, 0)]
    out = torch.full((q_len, 1, DV), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((1, q_len), float("nan"), dtype=torch.float32, device="cuda")
    ws = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    scale = 1.0 / np.sqrt(DQK)
    P.hydra_attn_fwd_local(q, k, v, cu, 1, 1, DQK, DV, q_chunks, q_len, kv_chunks, keys, pairs, True, scale, out, lse,
                           None, None, 0, ws)
    assert P.hydra_poll_status(ws)[0] == 0
    # the same in fp64, a block of keys at a time
    block = 1 << 20
    s = torch.cat([q[:, 0].double() @ k[i:i + block, 0].double().T for i in range(0, keys, block)], 1) * scale
    s.masked_fill_(torch.arange(keys, device="cuda")[None] > torch.arange(keys - q_len, keys, device="cuda")[:, None],
                   -float("inf"))
    ref_l = s.logsumexp(1)
    w = torch.exp(s - ref_l[:, None])
    ref_o = sum(w[:, i:i + block] @ v[i:i + block, 0].double() for i in range(0, keys, block))
    assert float((lse[0].double() - ref_l).abs().max()) <= TOL_LSE
    assert float((out[:, 0].double() - ref_o).abs().max()) <= TOL_REL * float(ref_o.abs().max())


@pytest.mark.parametrize("order", [(0, -1, 1280, -1), (0, 1280, -1, 1280)])
def test_a_limit_set_to_the_library_s_own_value_is_kept_to(order):
    """A 3000-token call of two heads has fewer tiles than SMs: the library sends it to the short-sequence kernel, halved.
    A caller who sets the limit, to 1280 like the library, keeps it on CTA pairs, whichever of the two came first."""
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import AttnStep, bits_to_tensor
    h, T = 2, 3000 + (order[1] < 0)                      # (a shape per order: no tables from the other one)
    cu = hw.cu_seqlens([T])
    x = rand_inputs(T, T, h)
    step = AttnStep(cu, h)
    q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
    got = {}
    for limit in order:
        P.hydra_set_fwd_short_len(limit)
        step.forward(q, k, v)
        assert step.poll()[0] == 0
        bits = step.out.view(torch.uint8).clone()
        assert limit not in got or torch.equal(bits, got[limit]), limit
        got[limit] = bits
    assert torch.equal(got[1280], got[0]), "not the CTA-pair kernel's result"
    assert not torch.equal(got[-1], got[0]), "the two kernels' sums differ in their last bits"


@pytest.mark.parametrize("length,copies", [(1100, 90), (1536, 45), (1537, 45)])   # tiles of up to 18, 24 and 25 steps
def test_many_copies_of_a_sequence_give_the_same_bits(length, copies):
    """In a call of many tiles of up to 24 steps the slots pop two items ahead, beyond that late: every copy of a sequence
    comes out as every other, and as the oracle has the first."""
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import AttnStep, bits_to_tensor
    P.hydra_set_fwd_short_len(1 << 20)
    x = rand_inputs(length, length, 2)
    step = AttnStep(hw.cu_seqlens([length] * copies), 2)
    step.out.fill_(float("nan"))
    step.lse.fill_(float("nan"))
    step.forward(*(bits_to_tensor(x[n]).repeat(copies, 1, 1) for n in ("q", "k", "v")))
    assert step.poll()[0] == 0
    out = step.out.view(torch.int16).view(copies, length, 2, DV)
    lse = step.lse.view(torch.int32).view(2, copies, length)
    assert bool((out == out[:1]).all()) and bool((lse == lse[:, :1]).all())
    ref = run_oracle(x, hw.cu_seqlens([length]), backward=False)
    got = dict(out=step.out[:length].float().cpu().numpy().astype(np.float64),
               lse=step.lse[:, :length].cpu().numpy().astype(np.float64))
    check(got, ref, names=("out", "lse"))


def test_random_length_mixes_and_both_kernels_agree():
    import paper_2609_34318_b200 as P
    rng = np.random.default_rng(11)
    for trial in range(4):
        lengths = [int(v) for v in rng.integers(1, 700, size=int(rng.integers(3, 12)))]
        h = int(rng.integers(1, 5))
        cu = hw.cu_seqlens(lengths)
        x = rand_inputs(100 + trial, int(cu[-1]), h)
        ref = run_oracle(x, cu, backward=False)
        res = {}
        for name, limit in (("short", 1 << 20), ("pair", 0)):
            P.hydra_set_fwd_short_len(limit)
            res[name] = run_gpu(x, cu, h, backward=False)
            check(res[name], ref, names=("out", "lse"), label=f"trial {trial} {name} ")
        # two summation orders of the same sums: a few bf16 roundings of O apart, never more
        assert np.abs(res["short"]["out"] - res["pair"]["out"]).max() <= TOL_REL * np.abs(ref["out"]).max()
        assert np.abs(res["short"]["lse"] - res["pair"]["lse"]).max() <= TOL_LSE


def test_one_call_uses_both_kernels_when_short_pairs_carry_enough_work():
    """A long sequence and many short ones: the long pair runs on CTA pairs, the short ones on the other kernel,
    in the same call (two launches); with few short ones the call stays on one kernel (one launch)."""
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import AttnStep, bits_to_tensor
    h = 2
    for lengths, launches in (([3000] + [300] * 60, 2), ([3000, 300, 300], 1), ([300] * 8, 1)):
        cu = hw.cu_seqlens(lengths)
        x = rand_inputs(len(lengths), int(cu[-1]), h)
        step = AttnStep(cu, h)
        q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
        assert forward_launches(lambda: step.forward(q, k, v)) == launches, lengths[:3]
        got = run_gpu(x, cu, h, backward=False)
        check(got, run_oracle(x, cu, backward=False), names=("out", "lse"), label=f"{lengths[:3]} ")


def test_a_limit_set_by_the_caller_is_kept_to_by_a_few_longer_pairs_too():
    """With the library's own limit a few pairs of up to twice its length stay on the short-sequence kernel, for the sake of
    one launch; a caller's limit sends every longer pair to CTA pairs."""
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import AttnStep, bits_to_tensor
    h, lengths = 2, [200] * 80 + [500] * 20              # 480 q tiles: not a call for halved ones
    cu = hw.cu_seqlens(lengths)
    x = rand_inputs(3, int(cu[-1]), h)
    step = AttnStep(cu, h)
    q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
    for limit, launches in ((256, 2), (499, 2), (500, 1), (FWD_SHORT_LEN_DEFAULT, 1), (0, 1)):
        P.hydra_set_fwd_short_len(limit)
        assert forward_launches(lambda: step.forward(q, k, v)) == launches, limit
        if limit == 256:
            check(run_gpu(x, cu, h, backward=False), run_oracle(x, cu, backward=False), names=("out", "lse"))


@pytest.mark.parametrize("h", [2, 10])                 # 20 q tiles a head: halved tiles, and more tiles than SMs
def test_chunked_short_pairs_write_partials_and_merge(h):
    """Short sequences cut into zigzag chunks: diagonal and full pairs with offsets, partial outputs, the merge."""
    lengths = [300, 77, 512, 130]
    cu = hw.cu_seqlens(lengths)
    x = rand_inputs(5, int(cu[-1]), h)
    lib_pairs, rows, ora_pairs = pairs_for(cu, [1, 0, 2, 1])
    got = run_gpu(x, cu, h, lib_pairs, rows)
    check(got, run_oracle(x, cu, pairs=ora_pairs), label="chunked short ")


@pytest.mark.parametrize("h", [2, 30])                 # 5 q tiles a head
def test_non_causal_short_pairs(h):
    lengths = [100, 65, 257]
    cu = hw.cu_seqlens(lengths)
    x = rand_inputs(6, int(cu[-1]), h)
    got = run_gpu(x, cu, h, causal=False)
    check(got, run_oracle(x, cu, causal=False), label="non-causal short ")


@pytest.mark.parametrize("short_len,h", [(FWD_SHORT_LEN_DEFAULT, 2), (FWD_SHORT_LEN_DEFAULT, 38), (0, 2)])   # 4 q tiles a head
def test_output_that_is_16_but_not_32_byte_aligned(short_len, h):
    """The interface asks for 16-byte alignment; both forward kernels store 32 bytes at a time only when the
    address allows it."""
    import paper_2609_34318_b200 as P
    P.hydra_set_fwd_short_len(short_len)
    from paper_2609_34318_b200.runner import AttnStep, bits_to_tensor
    lengths = [70, 300]
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    x = rand_inputs(7, T, h)
    step = AttnStep(cu, h)
    raw = torch.zeros(T * h * DV * 2 + 64, dtype=torch.uint8, device="cuda")
    off = (16 - raw.data_ptr() % 32) % 32                # an address that is 16 modulo 32
    out = raw[off:off + T * h * DV * 2].view(torch.bfloat16).view(T, h, DV)
    assert out.data_ptr() % 32 == 16
    q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
    P.hydra_attn_fwd(q, k, v, cu, h, None, True, step.scale, out, step.lse, None, None, 0, step.workspace)
    assert step.poll()[0] == 0
    ref = run_oracle(x, cu, backward=False)
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.abs(got - ref["out"]).max() <= TOL_REL * np.abs(ref["out"]).max()
    assert bool((raw[:off] == 0).all()) and bool((raw[off + T * h * DV * 2:] == 0).all())


@pytest.mark.parametrize("short_len,few_tiles", [(1 << 20, True), (1 << 20, False), (0, True)])
@pytest.mark.parametrize("q_start,q_len,k_start,k_len", [
    (0, 300, 200, 100),       # the first 200 q rows come before every key: a whole tile without keys, one with some
    (10, 140, 149, 60),       # only the last q row sees a key (its own position)
    (0, 130, 200, 90),        # no q row sees any key
    (50, 200, 0, 0),          # an empty kv range
    (255, 5, 0, 260),         # five rows at the end of a long kv range
])
def test_partials_of_hand_made_pairs_with_rows_that_see_no_key(short_len, few_tiles, q_start, q_len, k_start, k_len):
    """Rows of a pair that see no key get O = 0 and LSE = -inf (their weight in a merge is then 0): on both
    forward kernels, for whole tiles without keys, for single rows, and for pairs with no visible key at all. (With no
    more q tiles than SMs the short-sequence kernel shares every tile between two slots.)"""
    import oracle
    import paper_2609_34318_b200 as P
    from paper_2609_34318_b200.runner import AttnStep, bits_to_tensor
    P.hydra_set_fwd_short_len(short_len)
    lengths, h = [31, 300, 64], 2
    if not few_tiles:
        h = torch.cuda.get_device_properties(0).multi_processor_count // ((q_len + 127) // 128) + 1
    cu = hw.cu_seqlens(lengths)
    T = int(cu[-1])
    x = rand_inputs(q_start + k_len, T, h)
    pair = dict(seq=1, q_start=q_start, q_len=q_len, k_start=k_start, k_len=k_len, part_row=3, group=0)
    step = AttnStep(cu, h, [pair], q_len + 5)
    step.o_part.fill_(float("nan"))
    step.lse_part.fill_(float("nan"))
    q, k, v = (bits_to_tensor(x[n]) for n in ("q", "k", "v"))
    P.hydra_attn_fwd(q, k, v, cu, h, step.pairs, True, step.scale, step.out, step.lse, step.o_part, step.lse_part,
                     q_len + 5, step.workspace)
    assert step.poll()[0] == 0
    ref_o, ref_l = oracle.attn_partial(x["q"], x["k"], x["v"], cu, pair, True, np.float32(step.scale))
    got_o = step.o_part.float().cpu().numpy().astype(np.float64)
    got_l = step.lse_part.cpu().numpy().astype(np.float64)
    assert np.isnan(got_l[:, :3]).all() and np.isnan(got_l[:, 3 + q_len:]).all(), "rows outside the pair were written"
    o, l = got_o[3:3 + q_len], got_l[:, 3:3 + q_len]
    assert np.array_equal(np.isneginf(l), np.isneginf(ref_l)), "which rows see no key"
    fin = np.isfinite(ref_l)
    if fin.any():
        assert np.abs(l[fin] - ref_l[fin]).max() <= TOL_LSE
    assert np.abs(o - ref_o).max() <= TOL_REL * max(np.abs(ref_o).max(), 1e-30) + 0.0
    assert (o[np.isneginf(ref_l).T] == 0).all()
