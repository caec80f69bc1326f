"""GPU parity of the float64-accurate tensor-core likelihood (RIFT_FP64) at the edges of its
layouts: detectors, padded mode widths kp = 16, 32, 48, its limit of 42 components (24 modes
take the plain float64 kernel), time grids of one bin and around its 64-bin chunks, batches
around its 128-sample tiles, its unsorted small batches and the batches whose time bins are
split over blocks."""
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


LM24 = [(l, m) for l in range(2, 5) for m in range(-l, l + 1)] + [(5, -5), (5, 0), (5, 5)]

SHAPES = [
    # detectors, modes, sampling rate, time bins
    (("H1",), 1, 4096.0, 1),
    (("H1", "L1"), 2, 4096.0, 63),
    (("H1", "L1", "V1"), 8, 16384.0, 64),
    (("H1",), 9, 4096.0, 65),
    (("H1", "L1", "V1", "X1"), 16, 4096.0, 257),
    (("H1", "L1"), 17, 16384.0, 401),
    (("H1", "L1", "V1"), 21, 16384.0, 1001),
    (("H1", "L1"), LM24, 4096.0, 129),
]
COUNTS = [1, 127, 128, 129, 512, 513, 1500]


def problem(i, **more):
    dets, modes, fs, n_t = SHAPES[i]
    kw = dict(n_modes=modes) if isinstance(modes, int) else dict(lm=modes)
    return S.make_problem(dets, fs=fs, n_t=n_t, seed=S.config_seed(6, i), **kw, **more)


@pytest.mark.parametrize("i", range(len(SHAPES)))
@pytest.mark.parametrize("snr", [0.0, 20.0, 400.0])
def test_parity_and_independence_of_the_batch(G, oracle_lib, i, snr):
    """Every ln L and per-bin value against the float64 oracle.  Bound: positions carry
    2^-53 of ~3e3 Q samples (~4e-13) and a slope of at most the largest term per sample, the
    terms ~1e-15 of the largest: 1e-11 of the largest |ln L_t| of the sample.  A sample's
    value is the same bits in every batch."""
    p = problem(i, snr=snr)
    th = S.prior_samples(COUNTS[-1], 5)
    exp, ebins, _ = oracle_lib.lnL(p, th[:300], want_bins=True)
    scale = np.maximum(1.0, np.abs(ebins).max(axis=1))
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=COUNTS[-1]) as s:
        full, bins = s.eval(th, want_bins=True)
        assert np.all(np.abs(full[:300] - exp) <= 1e-11 * scale)
        assert np.all(np.abs(bins[:300] - ebins) <= 1e-11 * scale[:, None])
        for n in COUNTS[:-1]:
            assert np.array_equal(s.eval(th[-n:]), full[-n:])


def test_larger_than_the_split(G, oracle_lib):
    """A batch with more tiles than the split has records for (one bin range per tile) gives
    the same values as the same samples in small batches."""
    p = problem(3, snr=20.0)
    n = 4096 * 128 // 2 + 300
    th = S.prior_samples(n, 11)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
        full = s.eval(th)
        pick = np.random.default_rng(0).choice(n, 700, replace=False)
        assert np.array_equal(s.eval(th[pick]), full[pick])
    exp = oracle_lib.lnL(p, th[pick[:200]])
    assert np.all(np.abs(full[pick[:200]] - exp) <= 1e-11 * np.maximum(1.0, np.abs(exp).max()))


@pytest.mark.parametrize("col,code", [(0, "RIFT_ERANGE"), (2, "RIFT_ENONFINITE"), (5, "RIFT_ENONFINITE")])
@pytest.mark.parametrize("n", [1, 300])
def test_non_finite_samples(G, col, code, n):
    """A NaN sky angle has no Q index (RIFT_ERANGE), any other NaN no ln L (RIFT_ENONFINITE);
    the handle's next evaluation is unaffected."""
    p = problem(1, snr=20.0)
    th = S.prior_samples(n, 3)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=1000) as s:
        want = s.eval(th)
        bad = th.copy()
        bad[-1, col] = np.nan
        with pytest.raises(G.RiftError) as e:
            s.eval(bad)
        assert e.value.code == getattr(G, code)
        assert np.array_equal(s.eval(th), want)


@pytest.mark.parametrize("n,seed,few", [(20000, 4, True), (200000, 6, False)])
def test_mixed_re_evaluation_is_the_float64_value(G, n, seed, few):
    """RIFT_MIXED: the samples that carry weight have the float64 mode's ln L: to the last bit from
    the tensor-core kernel, which takes lists of more than 512 samples, to float64 rounding (the
    bound above) from the kernel of the short lists."""
    p = problem(5, snr=30.0 if few else 8.0)
    with G.ILE(p, precision=G.RIFT_MIXED, max_samples=n, seed=seed) as s:
        s.marginalize(n)
        th, _, ll, lw = s.last_batch(n)
    assert (np.count_nonzero(lw >= lw.max() - 40.0) <= 512) == few
    keep = lw >= lw.max() - 39.0
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
        want, bins = s.eval(th[keep][:4000], want_bins=True)
    if few:
        assert np.all(np.abs(want - ll[keep]) <= 1e-11 * np.maximum(1.0, np.abs(bins).max(axis=1)))
    else:
        assert np.array_equal(want, ll[keep][:4000])
