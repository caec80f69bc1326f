"""Small batches of the float64 mode, whose tiles are a quarter of the lanes while every (tile, chunk
of bins) has a block of its own, and whose last unit of a tile merges the chunks: around the sizes
where the tiles, the split and the merging kernel change, a sample's value is the bits that it has
in a large batch, call after call, and beside flagged samples."""
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


@pytest.mark.parametrize("dets,modes,n_t", [(("H1",), 1, 1), (("H1",), 3, 64), (("H1", "L1"), 2, 101),
                                            (("H1", "L1", "V1"), 9, 401), (("H1", "L1"), 21, 1100)])
def test_small_batches(G, dets, modes, n_t):
    p = S.make_problem(dets, modes, 4096.0, n_t=n_t, snr=20.0, seed=S.config_seed(6, 180 + modes))
    chunks = min(16, (n_t + 63) // 64)
    last = 32 * (152 // chunks)      # the largest batch of small tiles on 152 multiprocessors
    counts = sorted({1, 31, 32, 33, 96, 127, 129, 511, 513, last - 1, last, last + 1, last + 33})
    n = counts[-1] + 500
    th = S.prior_samples(n, 181)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
        full, bins = s.eval(th, want_bins=True)
        for c in counts:
            a, b = s.eval(th[:c], want_bins=True)
            assert np.array_equal(a, full[:c]) and np.array_equal(b, bins[:c])
            assert np.array_equal(s.eval(th[-c:]), full[-c:])
        bad = th[:97].copy()
        bad[40, 0] = np.nan
        for _ in range(2):
            with pytest.raises(G.RiftError):
                s.eval(bad)
            assert np.array_equal(s.eval(th[:97]), full[:97])
    # a handle whose scratch holds few blocks
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=97) as s:
        for c in (1, 33, 97):
            assert np.array_equal(s.eval(th[:c]), full[:c])


@pytest.mark.parametrize("n_t,n", [(1001, 20011), (65, 17000), (401, 90001)])
def test_planned_batches(G, n_t, n):
    """Large batches of wide delays, whose units are planned by the tiles' widths: split time grids
    and whole tiles (too many for the split's records)."""
    p = S.make_problem(("H1", "L1", "V1"), 4, 16384.0, n_t=n_t, snr=20.0, seed=S.config_seed(6, 190))
    th = S.prior_samples(n, 191)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
        full = s.eval(th)
        a = G.rift_ile_kernel_launches(s.h)
        assert np.array_equal(s.eval(th), full)
        assert G.rift_ile_kernel_launches(s.h) - a == 10   # keys, two passes of three, plan, likelihood, merge
        pick = np.random.default_rng(0).choice(n, 600, replace=False)
        assert np.array_equal(s.eval(th[pick]), full[pick])
