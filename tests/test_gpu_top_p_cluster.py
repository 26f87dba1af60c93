"""seq_tree_top_p_filter at the sizes where its clusters change: vocabularies around the smallest slice (4096 tokens), the
largest (16384) and the largest cluster (8 slices, beyond which one CTA takes the row), row counts that change the number of
CTAs per row, vocabularies that do not end on a group of four, cuts in each round of the histogram, in place and not.  The
nucleus is checked token by token: it must be the shortest prefix, in the exact order, that reaches top_p (fp64 masses; a
cut within 3e-6 of the mass may fall one token off, as everywhere in the tests of this call)."""
import numpy as np
import pytest
import torch

from paper_2402_12374_b200 import binding as B

pytestmark = pytest.mark.gpu


def _check(x, T, top_p, in_place):
    d = torch.device("cuda:0")
    rows, V = x.shape
    buf = torch.full((rows, (V + 3) // 4 * 4), 7.0, device=d)
    buf[:, :V] = torch.from_numpy(x).to(d)
    src = buf[:, :V]
    out = src if in_place else torch.full_like(buf, 9.0)[:, :V]
    kept = torch.full((rows,), -1, dtype=torch.int32, device=d)
    st = torch.zeros(1, dtype=torch.int32, device=d)
    B.seq_tree_top_p_filter(src, T, top_p, out=out, kept_out=kept, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    got, kept = out.cpu().numpy(), kept.cpu().numpy()
    assert (buf[:, V:].cpu().numpy() == 7.0).all()  # the padding is not the call's to write
    for r in range(rows):
        order = np.argsort(-x[r].astype(np.float64), kind="stable")
        p = np.exp((x[r][order].astype(np.float64) - x[r].max()) / T)
        cum = np.cumsum(p) / p.sum()
        n = int(kept[r])
        inside = np.isfinite(got[r])
        assert inside.sum() == n >= 1 and inside[order[:n]].all(), r     # a prefix of the exact order
        assert (got[r][inside] == x[r][inside]).all()
        assert cum[n - 1] >= top_p - 3e-6 and (n == 1 or cum[n - 2] < top_p + 3e-6), (r, n, cum[n - 1])


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("rows,V", [(1, 5), (2, 4095), (2, 4096), (3, 4097), (40, 16384), (150, 16385), (300, 4099), (2, 32770), (1, 131072), (1, 131073)])
def test_slices_and_clusters(rows, V, in_place):
    x = (3 * np.random.default_rng(rows + V).standard_normal((rows, V))).astype(np.float32)
    _check(x, 0.9, 0.9, in_place)


@pytest.mark.parametrize("top_p", [1e-6, 0.3, 0.5, 0.7, 0.9, 0.9999])
def test_cuts_in_every_round_of_the_histogram(top_p):
    """One token with a tenth of the mass, the rest spread thin behind exponent arguments of 8, 15, 16, 30 and 36."""
    V = 20000
    rng = np.random.default_rng(3)
    rows = []
    for d in (8.0, 15.0, 16.0, 30.0, 36.0):
        x = np.full(V, -40.0, np.float32)
        x[rng.choice(V, 12000, replace=False)] = (-d * np.log(2.0) + 0.3 * rng.standard_normal(12000)).astype(np.float32)
        x[777] = 0.0
        rows.append(x)
    _check(np.stack(rows), 1.0, top_p, False)


@pytest.mark.parametrize("in_place", [False, True])
def test_many_tokens_in_the_cut_of_one_row_only(in_place):
    """A row of equal logits (one CTA takes it) between ordinary ones."""
    rng = np.random.default_rng(8)
    x = (3 * rng.standard_normal((3, 30000))).astype(np.float32)
    x[1] = 0.25
    _check(x, 1.0, 0.6, in_place)


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("rows,V,spread", [(2, 128256, 0.5), (40, 50257, 0.2), (160, 16384, 0.05), (1, 131072, 0.01), (3, 128255, 1e-3), (2, 32770, 1e-5),
                                           (5, 4097, 0.0), (3, 600, 1e-3)])
def test_many_tokens_in_the_cut(rows, V, spread, in_place):
    """Rows whose cut's bin holds more tokens than are ordered at once, from a few hundred to the whole row (the bins' counters
    wrap from 4096 tokens per CTA on), cut at several places."""
    rng = np.random.default_rng(rows + V)
    x = (1.7 + spread * rng.standard_normal((rows, V))).astype(np.float32)
    for top_p in (0.9,) if V > 60000 else (1e-5, 0.37, 0.9, 0.99999):
        _check(x, 0.6, top_p, in_place)


@pytest.mark.parametrize("levels", [1, 2, 7, 300])
@pytest.mark.parametrize("rows,V", [(1, 30000), (2, 131072), (300, 5001)])
def test_runs_of_equal_logits_are_kept_in_token_order(rows, V, levels):
    """Few distinct logits, of both signs: the cut falls inside a run that spreads over all CTAs of a cluster."""
    rng = np.random.default_rng(levels)
    x = (rng.integers(0, levels, (rows, V)).astype(np.float32) - levels // 2) / 64.0
    for top_p in (0.003, 0.5, 0.97):
        _check(x, 0.8, top_p, False)


def test_flat_rows_with_what_never_counts():
    """NaN, infinities and tokens below 2^-40 of the most probable one beside thousands in one bin."""
    d = torch.device("cuda:0")
    V = 60000
    x = torch.full((2, V), 0.5, device=d)
    x[:, ::3] = float("-inf")
    x[:, 1::6] = -100.0
    x[1, 2], x[1, 8] = float("nan"), float("inf")
    out, kept = torch.empty_like(x), torch.empty(2, dtype=torch.int32, device=d)
    st = torch.zeros(1, dtype=torch.int32, device=d)
    B.seq_tree_top_p_filter(x, 1.0, 0.25, out=out, kept_out=kept, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == B.SEQ_DEV_NONFINITE
    for r in range(2):
        live = torch.nonzero(x[r] == 0.5).flatten()
        n = -(-len(live) // 4)
        assert int(kept[r]) == n
        assert torch.equal(torch.nonzero(out[r] > float("-inf")).flatten(), live[:n])


def test_no_spread_of_a_row_costs_many_times_another():
    """378 rows of 128256 tokens: equal logits take about five times what ordinary rows take, narrow ones two to three times (185
    and 8 times when one CTA took such a row)."""
    d = torch.device("cuda:0")
    x = torch.randn((378, 128256), device=d)
    out = torch.empty_like(x)

    def ms(logits):
        best = float("inf")
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            B.seq_tree_top_p_filter(logits, 0.6, 0.9, out=out)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    ordinary = ms(x * 3)
    for spread, times in ((0.0, 20), (0.05, 5)):
        assert ms(x * spread) < times * ordinary, spread


@pytest.mark.parametrize("spread,top_p", [(3.0, 0.9), (0.5, 0.37), (0.0, 0.6), (1e-3, 0.97)])
@pytest.mark.parametrize("V", [131073, 151936])
def test_rows_larger_than_a_cluster(V, spread, top_p):
    """One CTA per row, with and without the radix select."""
    x = (0.3 + spread * np.random.default_rng(V).standard_normal((3, V))).astype(np.float32)
    _check(x, 0.8, top_p, V == 151936)


def test_rows_larger_than_a_cluster_keep_enough_loads_in_flight():
    """A row of 131073 tokens on one CTA of 1024 threads takes about 72 us; on 512 threads it took 104."""
    d = torch.device("cuda:0")
    x = 3 * torch.randn((64, 131076), device=d)[:, :131073]
    x, out = torch.empty((64, 131076), device=d)[:, :131073].copy_(x), torch.empty((64, 131076), device=d)[:, :131073]
    best = float("inf")
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(5):
            B.seq_tree_top_p_filter(x, 0.6, 0.9, out=out)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) / 5 * 1e3)
    assert best < 100


@pytest.mark.parametrize("rows", [30, 31, 34, 35, 42, 43, 53, 54, 70, 71, 92, 93, 148])
def test_row_counts_that_change_the_clusters_side_by_side(rows):
    """Around the numbers of rows at which a row gets fewer CTAs because its clusters would not all be placed: every row as it
    comes out alone, bit for bit (the masses are integers, so the number of CTAs does not enter the result)."""
    d = torch.device("cuda:0")
    g = torch.Generator(device=d)
    g.manual_seed(rows)
    x = 3 * torch.randn((rows, 32000), device=d, generator=g)
    kept = torch.empty(rows, dtype=torch.int32, device=d)
    out = B.seq_tree_top_p_filter(x, 0.8, 0.9, kept_out=kept)
    for r in range(rows):
        one = torch.empty(1, dtype=torch.int32, device=d)
        assert torch.equal(B.seq_tree_top_p_filter(x[r:r + 1], 0.8, 0.9, kept_out=one), out[r:r + 1]) and int(one) == int(kept[r])
