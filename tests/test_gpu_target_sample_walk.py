"""Verification by sampling from the target on the walk with its rows in registers: vocabularies at the edges of a warp's
segment, of a CTA's slice and of what a thread holds, one node up to a full tree, and batches on clusters of 16 and of 8."""
import dataclasses

import pytest
import torch

from oracle import oracle as O
from paper_2402_12374_b200 import binding as B
from paper_2402_12374_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _inputs(V, n, seed, T=0.8):
    cfg = dataclasses.replace(W.CONFIGS["tiny"], n_tree=n, vocab=V, max_depth=8, max_fanout=5)
    vi = W.make_verify_inputs(cfg, T, seed)
    G.steer_tokens_to_samples(vi, every=2)  # deep walks
    return vi


@pytest.mark.parametrize("V,n", [(9, 4), (31, 9), (65, 20), (4097, 33), (32768, 40), (32769, 12), (65536, 10), (65537, 10), (131072, 6), (600, 1), (900, 1024)])
def test_one_request(V, n):
    outcomes = [G.check_verify_target_sample(_inputs(V, n, seed)) for seed in range(4)]
    assert outcomes.count("ok") >= 2  # (a draw inside the rounding band of a boundary is excluded)


@pytest.mark.parametrize("R,V,n", [(4, 1000, 20), (12, 500, 30), (10, 16385, 9), (40, 33, 17), (20, 65536, 5), (38, 65540, 3)])
def test_batch(R, V, n):
    d = G.dev()
    pad = (V + 3) // 4 * 4
    vis = [_inputs(V, n, 90 + r) for r in range(R)]
    tl = torch.full((R, n, pad), float("nan"), device=d)[..., :V]
    for r, vi in enumerate(vis):
        tl[r] = vi.target_logits.to(d)
    st = torch.zeros(1, dtype=torch.int32, device=d)
    path, plen, bonus = B.seq_tree_verify_batch(torch.stack([v.parent for v in vis]).to(d), torch.stack([v.tokens for v in vis]).to(d), tl, tl, 0.8,
                                                torch.stack([v.uniforms for v in vis]).to(d), dev_status=st, target_sample=True)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    clear = 0
    for r, vi in enumerate(vis):
        ref = O.tree_verify_target_sample(vi.parent, vi.tokens, vi.target_logits, 0.8, vi.uniforms)
        if ref["min_gap"] < G.GAP:
            continue
        clear += 1
        assert path[r, :int(plen[r])].cpu().tolist() == ref["path"].tolist() and int(bonus[r]) == ref["bonus"], r
    assert clear >= R // 2
