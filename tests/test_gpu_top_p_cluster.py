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
