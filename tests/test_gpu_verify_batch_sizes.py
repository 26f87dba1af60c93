"""seq_tree_verify_batch where the kernel that serves it changes: ten and more requests (clusters of 8 with rows in
registers), vocabularies at the edges of what a thread holds (16384, 32768, 65536 tokens, and one more), more requests of a
large vocabulary than the register walk takes, bfloat16 logits.  Every request against the oracle on it alone."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2402_12374_b200 import binding as B
from paper_2402_12374_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,V,n,mode,bf16", [(10, 32000, 24, "sequoia", False), (40, 1000, 12, "specinfer", False), (11, 16385, 10, "sequoia", False),
                                             (10, 32768, 12, "specinfer", False), (12, 32769, 12, "sequoia", False), (10, 50257, 10, "sequoia", True),
                                             (10, 65536, 9, "sequoia", False), (10, 65537, 9, "sequoia", False), (8, 40000, 9, "sequoia", False),
                                             (38, 65540, 3, "sequoia", False), (20, 33, 17, "sequoia", False)])
def test_large_batches(R, V, n, mode, bf16):
    d = G.dev()
    pad = (V + 3) // 4 * 4
    cfg = dataclasses.replace(W.CONFIGS["tiny"], n_tree=n, vocab=V, max_depth=6, max_fanout=4)
    T = 0.7
    vis = [W.make_verify_inputs(cfg, T, 50 + r) for r in range(R)]
    dt = torch.bfloat16 if bf16 else torch.float32
    tl = torch.full((R, n, pad), float("nan"), dtype=dt, device=d)[..., :V]
    dl = torch.full((R, n, pad), float("nan"), dtype=dt, device=d)[..., :V]
    for r, vi in enumerate(vis):
        tl[r], dl[r] = vi.target_logits.to(dt).to(d), vi.draft_logits.to(dt).to(d)
    resid = torch.full((R, V), float("nan"), dtype=torch.float32, device=d)
    nxt = torch.full((R, n), -9, dtype=torch.int32, device=d)
    st = torch.zeros(1, dtype=torch.int32, device=d)
    path, plen, bonus = B.seq_tree_verify_batch(torch.stack([v.parent for v in vis]).to(d), torch.stack([v.tokens for v in vis]).to(d), tl, dl, T,
                                                torch.stack([v.uniforms for v in vis]).to(d), residual_out=resid, next_child_out=nxt,
                                                dev_status=st, specinfer=mode == "specinfer")
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    clear = 0
    for r, vi in enumerate(vis):
        ref = O.tree_verify(vi.parent, vi.tokens, vi.target_logits.to(dt).float(), vi.draft_logits.to(dt).float(), T, vi.uniforms,
                            variant=O.VARIANT_SPECINFER if mode == "specinfer" else O.VARIANT_SEQUOIA)
        if ref["min_gap"] < G.GAP:
            continue
        clear += 1
        k = int(plen[r].item())
        assert path[r, :k].cpu().tolist() == ref["path"].tolist(), r
        want = np.full(n, -2)
        want[ref["path"][:-1]] = ref["path"][1:]
        want[ref["path"][-1]] = -1
        assert np.array_equal(nxt[r].cpu().numpy(), want)
        got = resid[r].double().cpu().numpy()
        assert np.abs(got - ref["residual"]).max() < G.RESID_TOL
        t, u, cdf = int(bonus[r].item()), float(vi.uniforms[n]), np.cumsum(ref["residual"])
        assert ref["residual"][t] > 0 and (t == 0 or cdf[t - 1] - 1e-5 <= u) and u < cdf[t] + 1e-5
    assert clear >= R - 2


@pytest.mark.parametrize("R", [37, 38, 60])
def test_bf16_batches_beyond_what_the_shared_memory_walk_would_take(R):
    """From 38 requests (148 SMs) a vocabulary above 65536 is the shared-memory walk's in fp32; it has no 16-bit form."""
    test_large_batches(R, 65540, 3, "sequoia", True)
