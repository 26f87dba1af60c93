"""Attention at the sizes where a tile can go wrong, every output against the oracle: groups of heads that do not divide a
tile of 128 rows on the tensor cores, and the single-precision kernel at the edges of its row tiles (8, 16, 32, 64 rows),
of its groups of 32 keys and of its key-range splits."""
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


@pytest.mark.parametrize("kernel", [B.KERNEL_AUTO, B.KERNEL_TENSOR_CORE_STREAM, B.KERNEL_TENSOR_CORE_GRID])
@pytest.mark.parametrize("hkv,group,n,L", [(1, 3, 42, 33), (1, 3, 43, 0), (2, 5, 25, 64), (2, 5, 101, 150), (1, 6, 1, 20), (2, 7, 36, 300),
                                           (1, 12, 25, 63), (1, 100, 3, 50), (1, 127, 2, 65)])
def test_groups_that_do_not_divide_the_tile(hkv, group, n, L, kernel):
    G.check_attention(_inputs(hkv, group, n, L, "bf16"), kernel=kernel)


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("kernel", [B.KERNEL_AUTO, B.KERNEL_TENSOR_CORE_STREAM, B.KERNEL_TENSOR_CORE_GRID])
@pytest.mark.parametrize("hkv,group,n,L", [(2, 5, 30, 700), (1, 3, 50, 150), (1, 12, 25, 63), (1, 100, 3, 1200)])
def test_probabilities_are_not_rounded_once_for_groups_that_do_not_divide_the_tile(hkv, group, n, L, dtype, kernel):
    """The output is no further from fp64 than its own rounding puts it.  P as two pieces is off by 2^-17 at most (bfloat16;
    half 2^-22), far below the output's 2^-9 (2^-12): 2 % of margin covers it.  P rounded once is off by as much as the
    output is, independently: 25 to 40 % more."""
    ai = _inputs(hkv, group, n, L, dtype)
    out, _, status = G.run_attention(ai, kernel)
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache, ai.v_cache, ai.parent, L)
    rounded = torch.from_numpy(ref).to(ai.q.dtype).double().numpy()
    assert status == 0
    assert np.linalg.norm(out.double().cpu().numpy() - ref) < 1.02 * np.linalg.norm(rounded - ref)


@pytest.mark.parametrize("hkv,n,L", [(60, 2, 1250), (40, 3, 1100), (32, 2, 1030), (24, 3, 1590), (16, 4, 3000), (1, 5, 2200), (1, 4, 4000)])
def test_clusters_of_every_size(hkv, n, L):
    """Where the device runs 74, 44, 36, 28, 21, 14 and 14 clusters of 2 to 8 CTAs side by side, these take one size each."""
    G.check_attention(_inputs(hkv, 1, n, L, "bf16"))


def _launched_cluster_size(hkv, n, L):
    """CTAs along the key range of the attention's launch, read off a captured graph (the grid's z extent)."""
    from cuda.bindings import driver

    d = G.dev()
    ai = _inputs(hkv, 1, n, L, "bf16")
    call = B.AttentionCall(ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d), None, L, parent=ai.parent.to(d))
    call.run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call.run()
    raw = driver.CUgraph(graph.raw_cuda_graph())
    _, _, count = driver.cuGraphGetNodes(raw)
    assert count == 1
    rc, nodes, _ = driver.cuGraphGetNodes(raw, count)
    assert rc == driver.CUresult.CUDA_SUCCESS
    rc, params = driver.cuGraphKernelNodeGetParams(nodes[0])
    assert rc == driver.CUresult.CUDA_SUCCESS
    return params.gridDimZ


def test_the_shapes_above_take_clusters_of_every_size():
    """Should the plan's constants or the device's occupancy move, the test above would go on passing without its purpose."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the shapes are chosen for 148 SMs")
    sizes = [_launched_cluster_size(*shape) for shape in [(60, 2, 1250), (40, 3, 1100), (32, 2, 1030), (24, 3, 1590), (16, 4, 3000), (1, 5, 2200), (1, 4, 4000)]]
    assert set(sizes) == set(range(2, 9)), sizes


@pytest.mark.parametrize("hkv,group,n,L", [(1, 1, 1, 0), (2, 1, 8, 31), (1, 1, 9, 119), (1, 2, 8, 128), (2, 3, 11, 97), (1, 1, 32, 96), (1, 1, 33, 224),
                                           (2, 4, 16, 255), (1, 5, 13, 64), (3, 1, 65, 63), (1, 150, 2, 40), (1, 1, 1, 3000)])
def test_single_precision_tiles(hkv, group, n, L):
    G.check_attention(_inputs(hkv, group, n, L, "fp32"))


def test_single_precision_with_the_length_in_device_memory():
    """Rows behind the tree hold NaN: they are fetched in this mode and must not reach a result."""
    d = G.dev()
    n, L, slack = 21, 75, 60
    ai = _inputs(2, 3, n, L, "fp32")
    pad = torch.full((2, slack, 128), float("nan"))
    k, v = (torch.cat([t[:, :L + n], pad], dim=1).contiguous().to(d) for t in (ai.k_cache, ai.v_cache))
    mask, _, st = G.gpu_mask(ai.parent.numpy())
    out = B.seq_tree_attention(ai.q.to(d), k, v, mask, L + slack - 1, dev_status=st, prefix_len_dev=torch.tensor([L], dtype=torch.int32, device=d))
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache[:, :L + n], ai.v_cache[:, :L + n], ai.parent, L)
    assert np.abs(out.double().cpu().numpy() - ref).max() < 1e-5


@pytest.mark.parametrize("hkv,group,n,L", [(8, 5, 100, 500), (32, 1, 64, 1024)])
def test_single_precision_sums_over_keys_stay_short(hkv, group, n, L):
    """Relative error against fp64 below six units of 2^-24.  A score's two chains of 64 products leave about four (the same
    whatever the prefix), 32-key sums and their few additions one; one chain over 600 or 1088 keys adds three and more."""
    ai = _inputs(hkv, group, n, L, "fp32")
    out, _, status = G.run_attention(ai)
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache, ai.v_cache, ai.parent, L)
    assert status == 0
    assert np.linalg.norm(out.double().cpu().numpy() - ref) < 6 * 2.0 ** -24 * np.linalg.norm(ref)


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("hkv,group,n,L", [(2, 1, 40, 70), (2, 3, 9, 0), (1, 1, 5, 3000), (1, 8, 70, 33)])
def test_single_precision_rows_do_not_depend_on_other_branches(hkv, group, n, L, bad):
    """A key and value row that holds infinities or NaN reaches the node's own row and its descendants', no other one."""
    d = G.dev()
    ai = _inputs(hkv, group, n, L, "fp32")
    parent = ai.parent.numpy()
    victim = 1
    sees = np.zeros(n, dtype=bool)
    for i in range(n):
        sees[i] = i == victim or (parent[i] >= 0 and sees[parent[i]])
    mask, _, _ = G.gpu_mask(parent)
    q, k, v = ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d)
    want = B.seq_tree_attention(q, k, v, mask, L).clone()
    k[:, L + victim], v[:, L + victim] = bad, bad
    got = B.seq_tree_attention(q, k, v, mask, L)
    torch.cuda.synchronize()
    assert 0 < sees.sum() < n
    assert torch.equal(got[~sees], want[~sees])
    assert not torch.isfinite(got[sees]).any()


@pytest.mark.parametrize("hkv,group,n,cap", [(2, 2, 8, 8192), (8, 8, 64, 8192), (8, 5, 100, 8192)])
def test_single_precision_workspace_of_the_longest_prefix_serves_every_shorter_one(hkv, group, n, cap):
    """The plan's own need rises and falls with the prefix length: every length of a decoding run, in steps of 32, is taken
    with the workspace of the longest one, and a few that would like more of it agree with the oracle."""
    d = G.dev()
    ai = _inputs(hkv, group, n, cap, "fp32")
    mask, _, _ = G.gpu_mask(ai.parent.numpy())
    q, k, v = ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d)
    longest = B.AttentionCall(q, k, v, mask, cap)
    short = 0
    for L in range(0, cap, 32):
        own = B.AttentionCall(q, k, v, mask, L, workspace=torch.empty(0, dtype=torch.uint8, device=d))
        call = B.AttentionCall(q, k, v, mask, L, workspace=longest.workspace)
        out = call.run()  # (refused: raises)
        if own.workspace_bytes_needed > longest.workspace_bytes_needed and short < 3:
            short += 1
            ref, _, _ = O.tree_attention(ai.q, ai.k_cache[:, :L + n], ai.v_cache[:, :L + n], ai.parent, L)
            assert np.abs(out.double().cpu().numpy() - ref).max() < 1e-5
    torch.cuda.synchronize()


def test_single_precision_without_a_workspace():
    """Shapes with rows for every SM never needed one; the split of the key range is then left out."""
    d = G.dev()
    ai = _inputs(32, 1, 64, 1000, "fp32")
    mask, _, _ = G.gpu_mask(ai.parent.numpy())
    call = B.AttentionCall(ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d), mask, 1000, workspace=torch.empty(0, dtype=torch.uint8, device=d))
    out = call.run()
    torch.cuda.synchronize()
    ref, _, _ = O.tree_attention(ai.q, ai.k_cache, ai.v_cache, ai.parent, 1000)
    assert np.abs(out.double().cpu().numpy() - ref).max() < 1e-5


@pytest.mark.parametrize("hkv,group,n,L", [(8, 5, 500, 4600), (50, 3, 126, 2100)])
def test_groups_that_do_not_divide_the_tile_without_a_workspace(hkv, group, n, L):
    """More tiles than SMs and many keys: the plan would like a workspace; without one the same tiles run one per CTA."""
    d = G.dev()
    ai = _inputs(hkv, group, n, L, "bf16")
    mask, _, st = G.gpu_mask(ai.parent.numpy())
    q, k, v = ai.q.to(d), ai.k_cache.to(d), ai.v_cache.to(d)
    call = B.AttentionCall(q, k, v, mask, L, workspace=torch.empty(0, dtype=torch.uint8, device=d), dev_status=st)
    assert call.workspace_bytes_needed > 0
    got, want = call.run(), B.seq_tree_attention(q, k, v, mask, L, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    rows = [0, 1, n // 2, n - 1]
    G.check_attention(ai, rows=rows)
    assert (got.float() - want.float()).abs().max() < 2e-2  # (both within half a unit of the exact rows, which are below 2)
    with pytest.raises(RuntimeError):
        B.AttentionCall(q, k, v, mask, L, workspace=torch.empty(0, dtype=torch.uint8, device=d), kernel=B.KERNEL_TENSOR_CORE_STREAM).run()
