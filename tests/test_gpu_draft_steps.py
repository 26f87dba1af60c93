"""seq_tree_draft_sample where its steps, parts and lists end: vocabularies around multiples of a step (4096 tokens) and of a
part, one to eight CTAs per row, up to 64 draws, rows whose best tokens all come last, rows of equal keys and rows with
fewer tokens in the running than draws (the list overflows or the threshold stays open).  Tokens against the oracle, rows
with keys closer than fp32 resolves left out as in the other tests of this call."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2402_12374_b200 import binding as B
from tests.test_gpu_draft_sample import _check_rows, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,V,k", [(3, 4095, 16), (3, 4096, 17), (3, 4097, 64), (2, 8192, 9), (150, 12289, 3), (60, 32769, 8), (500, 8193, 5),
                                      (1, 131072, 64), (2, 65541, 33)])
def test_vocabularies_at_the_edges_of_steps_and_parts(rows, V, k):
    rng = np.random.default_rng(V + k)
    logits = (3 * rng.standard_normal((rows, V))).astype(np.float32)
    u = rng.random((rows, V)).astype(np.float32)
    ok, excl, st = _check_rows(logits, u, 0.6, k)
    assert st == 0 and ok >= 0.7 * rows, (ok, excl)


@pytest.mark.parametrize("rows,V", [(1, 40000), (450, 9000)])
def test_rows_whose_best_tokens_come_last(rows, V):
    """Every step's tokens beat all earlier ones: the list overflows and the row is ranked 256 tokens at a time."""
    logits = np.tile(np.linspace(0.0, 400.0, V, dtype=np.float32), (rows, 1))
    u = np.full((rows, V), 0.5, np.float32)
    d = _dev()
    got = B.seq_tree_draft_sample(torch.from_numpy(logits).to(d), 0.5, torch.from_numpy(u).to(d), 64).cpu().numpy()
    assert (got == np.arange(V - 1, V - 65, -1)[None]).all()


@pytest.mark.parametrize("rows,V,k", [(1, 3000, 64), (2, 70000, 7), (450, 5000, 64)])
def test_equal_keys_go_in_token_order(rows, V, k):
    d = _dev()
    got = B.seq_tree_draft_sample(torch.zeros((rows, V), device=d), 1.0, torch.full((rows, V), 0.3, device=d), k).cpu().numpy()
    assert (got == np.arange(k)[None]).all()


@pytest.mark.parametrize("finite", [0, 1, 5, 40, 3000])
def test_rows_with_few_tokens_in_the_running(finite):
    rng = np.random.default_rng(finite)
    rows, V, k = 4, 30001, 40
    logits = np.full((rows, V), -np.inf, np.float32)
    for r in range(rows):
        logits[r, rng.choice(V, finite, replace=False)] = rng.standard_normal(finite)
    u = rng.random((rows, V)).astype(np.float32)
    d = _dev()
    got = B.seq_tree_draft_sample(torch.from_numpy(logits).to(d), 1.0, torch.from_numpy(u).to(d), k).cpu().numpy()
    for r in range(rows):
        ref = O.draft_sample(logits[r], 1.0, u[r], k)
        assert (got[r] >= 0).sum() == min(k, finite)
        if finite == 0 or ref["min_rel_gap"] >= 1e-4:
            assert got[r].tolist() == ref["tokens"].tolist()


@pytest.mark.parametrize("rows,V,k", [(378, 128256, 9), (300, 130000, 64), (9, 131072, 33)])
def test_rankings_between_steps_keep_every_listed_token(rows, V, k):
    """Rows of many steps, ranked after the 2nd, 4th, 8th, 16th and 32nd while warps that are ahead list the next step's
    tokens: the same tokens on every one of twenty calls, and those of a sort in double precision."""
    d = _dev()
    g = torch.Generator(device=d)
    g.manual_seed(k)
    logits = torch.randn((rows, V), device=d, generator=g) * 3
    u = torch.rand((rows, V), device=d, generator=g)
    first = B.seq_tree_draft_sample(logits, 0.6, u, k).clone()
    for _ in range(19):
        assert torch.equal(B.seq_tree_draft_sample(logits, 0.6, u, k), first)
    clear = 0
    for r in range(rows):
        score = logits[r].double() / float(np.float32(0.6)) - torch.log(-torch.log(u[r].double()))
        best = torch.topk(torch.where(u[r] > 0, score, torch.full_like(score, float("-inf"))), k + 1)
        if (best.values[:-1] - best.values[1:]).min() > 1e-4:
            clear += 1
            assert first[r].tolist() == best.indices[:k].tolist(), r
    assert clear >= rows // 2


@pytest.mark.parametrize("T", [1e-28, 1e-31, 1e-33, 1e-36, 2e-38])
def test_scores_of_any_magnitude(T):
    """At such temperatures the uniforms do not matter any more (logit / T in single precision swallows them): the draw is the
    order of the logits.  At 2e-38 the scores of the largest ones are infinite: equal, in token order."""
    rng = np.random.default_rng(5)
    rows, V, k = 64, 5000, 4
    logits = (3 * rng.standard_normal((rows, V))).astype(np.float32)
    u = (rng.random((rows, V)) * 0.9 + 0.05).astype(np.float32)
    d = _dev()
    got = B.seq_tree_draft_sample(torch.from_numpy(logits).to(d), T, torch.from_numpy(u).to(d), k).cpu().numpy()
    with np.errstate(over="ignore"):
        score = logits * (np.float32(1) / np.float32(T))
    want = np.argsort(-score, axis=1, kind="stable")[:, :k]
    assert (got == want).all()


@pytest.mark.parametrize("rows,V,k", [(3, 40000, 64), (2, 33333, 1), (450, 20001, 9), (5, 131072, 33)])
def test_lists_that_overflow_behind_ranked_steps(rows, V, k):
    """Equal uniforms, so that the draw is the order of the logits, lower token first: noise for a third of the row, then
    a staircase of runs of 37 equal logits that rises above it, the last third level with its top; the k-th token lies in
    a run.  A NaN behind the overflow is flagged."""
    rng = np.random.default_rng(V)
    logits = np.empty((rows, V), np.float32)
    third = V // 3
    logits[:, :third] = rng.standard_normal((rows, third))
    logits[:, third:] = 2.0 + np.minimum(np.arange(V - third), third) // 37 / 64.0
    want = np.argsort(-logits, axis=1, kind="stable")[:, :k]
    logits[0, V - 1] = np.nan
    d = _dev()
    st = torch.zeros(1, dtype=torch.int32, device=d)
    got = B.seq_tree_draft_sample(torch.from_numpy(logits).to(d), 0.7, torch.full((rows, V), 0.5, device=d), k, dev_status=st).cpu().numpy()
    assert (got == want).all()
    assert int(st.item()) == B.SEQ_DEV_NONFINITE


@pytest.mark.parametrize("order", ["equal", "ascending"])
def test_no_order_of_a_row_costs_many_times_another(order):
    """378 rows of 128256 tokens: two to four times the time of random rows (160 times when a list that overflowed was ranked 256
    tokens at a time)."""
    d = _dev()
    rows, V, k = 378, 128256, 9
    u = torch.rand((rows, V), device=d)
    half = torch.full((rows, V), 0.5, device=d)
    x = torch.zeros((rows, V), device=d) if order == "equal" else torch.linspace(0, 400, V, device=d).repeat(rows, 1)

    def ms(logits, uniforms):
        best = float("inf")
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            B.seq_tree_draft_sample(logits, 0.6, uniforms, k)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    assert ms(x, half) < 10 * ms(torch.randn((rows, V), device=d), u)
