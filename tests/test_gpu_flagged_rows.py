"""Per-bin values of a flagged sample in the float64 mode: NaN in every bin (never what the caller's
buffer held before), beside the values of the batch's other samples, with whole and split time
grids and for tiles without any finite sample."""
import numpy as np
import pytest

import ile_synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_11655_gb300 as G
    G.load(build_if_missing=True)
    return G


@pytest.mark.parametrize("n,bad", [(1, [0]), (300, [0, 131, 299]), (300, list(range(128, 256))), (9000, [17, 8999])])
@pytest.mark.parametrize("n_t", [1, 65, 401])
@pytest.mark.parametrize("col", [0, 2])
def test_rows(G, n, bad, n_t, col):
    import torch
    p = S.make_problem(("H1", "L1"), 3, 4096.0, n_t=n_t, snr=12.0, seed=S.config_seed(6, 140))
    th = S.prior_samples(n, 141)
    x = th.copy()
    x[bad, col] = np.nan
    keep = np.setdiff1d(np.arange(n), bad)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
        want, wbins = s.eval(th, want_bins=True)
        v = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
        rows = torch.full((n, n_t), 7.0, dtype=torch.float64, device="cuda")
        with pytest.raises(G.RiftError):
            G.rift_ile_eval(s.h, torch.from_numpy(x).cuda(), n, v, rows)
        v, rows = v.cpu().numpy(), rows.cpu().numpy()
    assert np.isnan(v[bad]).all() and np.isnan(rows[bad]).all()
    assert np.array_equal(v[keep], want[keep]) and np.array_equal(rows[keep], wbins[keep])
