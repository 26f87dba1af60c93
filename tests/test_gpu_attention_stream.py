"""The tensor-core attention's stream schedule where its two chains share an accumulator and a reference maximum, the outputs
that leave through shared memory, and the calls whose schedule depends on a workspace."""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2402_12374_b200 import binding as B
from paper_2402_12374_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _inputs(hkv, group, n, L, dtype, seed=3):
    cfg = dataclasses.replace(W.CONFIGS["tiny"], num_q_heads=hkv * group, num_kv_heads=hkv, prefix_len=L, n_tree=n, max_depth=14, max_fanout=8)
    return W.make_attention_inputs(cfg, seed, dtype=dtype, extra_capacity=9)


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("step", [64, 128, 192])
@pytest.mark.parametrize("hkv,group,n,L", [(2, 1, 30, 700), (1, 8, 20, 1000), (1, 5, 30, 450)])
def test_scores_that_rise_along_the_keys(hkv, group, n, L, step, dtype):
    """Every `step` keys the scores of all rows rise by 12 (17 in powers of two, beyond the 8 a reference lets pass): the
    reference moves in one chain's turn, in the other's, or in both, and the accumulator is rescaled.  The output is then all
    but decided by the last keys, to the output type's rounding of V (2e-2 covers four of bfloat16's)."""
    ai = _inputs(hkv, group, n, L, dtype)
    u = torch.ones(128) / 128 ** 0.5
    total = L + n
    rise = 12.0 * torch.floor(torch.arange(total) / step)
    q = (0.3 * ai.q.float() - (0.3 * ai.q.float() @ u)[..., None] * u + 16.0 * u).to(ai.q.dtype)
    k = ai.k_cache.float().clone()
    k[:, :total] = 0.3 * k[:, :total]
    k[:, :total] -= (k[:, :total] @ u)[..., None] * u
    k[:, :total] += (rise * 128 ** 0.5 / 16.0)[None, :, None] * u
    if dtype == "fp16" and float(k.abs().max()) > 6e4:
        pytest.skip("keys beyond half precision")
    ai = dataclasses.replace(ai, q=q, k_cache=k.to(ai.k_cache.dtype))
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache, ai.v_cache, ai.parent, L)
    for kernel in (B.KERNEL_TENSOR_CORE_STREAM, B.KERNEL_TENSOR_CORE_GRID):
        out, _, status = G.run_attention(ai, kernel)
        assert status == 0
        assert np.abs(out.double().cpu().numpy() - ref).max() < 2e-2


@pytest.mark.parametrize("hkv,group,n,L", [(1, 1, 1, 0), (1, 1, 1, 63), (1, 1, 1, 64), (1, 1, 3, 126), (1, 8, 17, 190), (2, 4, 33, 64), (3, 1, 129, 0),
                                           (1, 2, 65, 319), (8, 8, 40, 1500)])
def test_pairs_of_blocks(hkv, group, n, L):
    """One block, one pair, an odd block behind pairs, pieces of every size; mask given and derived from the tree."""
    ai = _inputs(hkv, group, n, L, "bf16")
    G.check_attention(ai, kernel=B.KERNEL_TENSOR_CORE_STREAM)
    d = G.dev()
    mask, _, st = G.gpu_mask(ai.parent.numpy())
    args = (ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d))
    given = B.seq_tree_attention(*args, mask, L, kernel=B.KERNEL_TENSOR_CORE_STREAM)
    derived = B.seq_tree_attention(*args, None, L, parent=ai.parent.to(d), kernel=B.KERNEL_TENSOR_CORE_STREAM, dev_status=st)
    assert torch.equal(given, derived) and int(st.item()) == 0


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("hkv,group,n,L", [(2, 5, 26, 1500), (2, 3, 43, 2000), (1, 5, 100, 3001), (3, 3, 128, 900)])
def test_groups_that_do_not_divide_a_tile_on_long_prefixes(hkv, group, n, L, dtype):
    """Their probabilities enter the product in two pieces, the second stored where scores of the same pair are read from: on
    unmasked pairs the output is as good as the exact one rounded to its type.  The two pieces leave 2^-16 (bfloat16) or 2^-22
    (half) of a probability at most, single precision less: a thirty-second of a unit in the last place covers them."""
    ai = _inputs(hkv, group, n, L, dtype)
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache, ai.v_cache, ai.parent, L)
    out, _, status = G.run_attention(ai, B.KERNEL_TENSOR_CORE_STREAM)
    assert status == 0
    rounded = torch.from_numpy(ref).to(out.dtype).double().numpy()
    unit = 2.0 ** (-7 if dtype == "bf16" else -10)
    assert np.linalg.norm(out.double().cpu().numpy() - ref) < np.linalg.norm(rounded - ref) + unit / 32 * np.linalg.norm(ref)


@pytest.mark.parametrize("kernel", [B.KERNEL_TENSOR_CORE_STREAM, B.KERNEL_TENSOR_CORE_GRID])
@pytest.mark.parametrize("hkv,group,n", [(1, 1, 80), (1, 1, 81), (2, 8, 10), (2, 8, 11), (1, 5, 17), (1, 1, 128), (1, 3, 43), (1, 1, 200)])
def test_outputs_with_strides_of_their_own(hkv, group, n, kernel):
    """Rows of the output apart from each other, around the number of rows from which they leave through shared memory;
    nothing between them is touched."""
    d, L = G.dev(), 20
    ai = _inputs(hkv, group, n, L, "fp16")
    mask, _, st = G.gpu_mask(ai.parent.numpy())
    Hq = hkv * group
    buf = torch.full((n, Hq + 1, 128 + 8), 7.0, dtype=torch.float16, device=d)
    out = buf[:, :Hq, :128]
    B.seq_tree_attention(ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d), mask, L, out=out, dev_status=st, kernel=kernel)
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache, ai.v_cache, ai.parent, L)
    assert int(st.item()) == 0
    assert np.abs(out.double().cpu().numpy() - ref).max() < G.ATTN_TOL[torch.float16]
    assert bool((buf[:, Hq] == 7.0).all()) and bool((buf[:, :, 128:] == 7.0).all())


def test_a_stream_that_is_only_the_faster_choice_needs_no_workspace():
    """96 units of 131 blocks: streamed where a workspace is lent, served by the grid schedule where none (or a short or
    misaligned one) is."""
    d = G.dev()
    n, L = 384, 8000
    ai = _inputs(8, 4, n, L, "bf16")
    parent = ai.parent.to(d)
    args = (ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d))
    call = B.AttentionCall(*args, None, L, parent=parent)
    streamed = call.run().clone()
    if torch.cuda.get_device_properties(d).multi_processor_count != 148:
        pytest.skip("the rule's figures are those of 148 SMs")
    assert call.workspace_bytes_needed > 0
    stream = B.seq_tree_attention(*args, None, L, parent=parent, kernel=B.KERNEL_TENSOR_CORE_STREAM)
    forced = B.seq_tree_attention(*args, None, L, parent=parent, kernel=B.KERNEL_TENSOR_CORE_GRID)
    assert torch.equal(streamed, stream) and not torch.equal(streamed, forced)
    assert (streamed.float() - forced.float()).norm() < 5e-3 * forced.float().norm()  # two roundings of P to bfloat16
    backing = torch.empty(call.workspace_bytes_needed + 256, dtype=torch.uint8, device=d)
    for lent in (backing[:0], backing[:4096], backing[8:8 + call.workspace_bytes_needed]):
        got = B.seq_tree_attention(*args, None, L, parent=parent, workspace=lent)
        assert torch.equal(got, forced)
    # with the length in device memory, which may be far below the bound that the launch is planned for, the grid schedule
    length = torch.tensor([L], dtype=torch.int32, device=d)
    replayed = B.AttentionCall(*args, None, L, parent=parent, prefix_len_dev=length)
    assert replayed.workspace_bytes_needed == 0 and torch.equal(replayed.run(), forced)


@pytest.mark.parametrize("kernel", [B.KERNEL_AUTO, B.KERNEL_TENSOR_CORE_STREAM])
@pytest.mark.parametrize("hq,hkv,n,bound", [(64, 8, 16, 20000), (32, 8, 16, 18432), (32, 4, 16, 13312), (8, 1, 3, 9000)])
def test_lengths_in_device_memory_far_below_the_bound(hq, hkv, n, bound, kernel):
    """A launch planned for a long prefix that meets a short one: the layout then has fewer positions than the grid has CTAs,
    and every tile is written all the same (the output starts as NaN)."""
    d = G.dev()
    ai = _inputs(hkv, hq // hkv, n, bound, "bf16")
    q, k, v, parent = ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d), ai.parent.to(d)
    st = torch.zeros(1, dtype=torch.int32, device=d)
    length = torch.zeros(1, dtype=torch.int32, device=d)
    out = torch.empty_like(q)
    call = B.AttentionCall(q, k, v, None, bound, parent=parent, out=out, dev_status=st, kernel=kernel, prefix_len_dev=length)
    for L in (0, 64, 100, 200, 300, 500, 600, 1000, bound):
        length.fill_(L)
        out.fill_(float("nan"))
        call.run()
        if L < bound:
            ref = O.tree_attention(ai.q, ai.k_cache[:, :L + n], ai.v_cache[:, :L + n], ai.parent, L)[0]
        else:  # (the oracle would take its time)
            ref = B.seq_tree_attention(q, k, v, None, L, parent=parent, kernel=B.KERNEL_TENSOR_CORE_GRID).double().cpu().numpy()
        err = np.abs(out.double().cpu().numpy() - ref).max()
        assert err < G.ATTN_TOL[torch.bfloat16], f"prefix {L}: {err}"  # (NaN is not below it)
    assert int(st.item()) == 0
