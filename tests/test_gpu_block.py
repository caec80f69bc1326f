"""GPU parity of the CUDA-core float32 likelihood (RIFT_ILE_TC=0) at the edges of its plan:
chunks of up to 1024 time bins in groups of 128, blocks of 4 and of 8 samples, unsorted and
sorted batches, windows that do not fit the R tile together (they are contracted in turn) or
need several chunks, and the distance marginal.  Float32 bar of the other parity checks:
|d ln L| <= 1e-3 on every sample and time bin."""
import numpy as np
import pytest

import ile_synth as S

pytestmark = pytest.mark.gpu
TOL = 1e-3


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_11655_gb300 as G
    G.load(build_if_missing=True)
    return G


SHAPES = [
    # detectors, modes, sampling rate, time bins
    (("H1",), 1, 4096.0, 1),
    (("H1", "L1"), 2, 4096.0, 31),
    (("H1", "L1", "V1"), 5, 4096.0, 129),
    (("H1", "L1", "V1", "X1"), 9, 4096.0, 1024),
    (("H1", "L1"), 3, 16384.0, 1025),
    (("H1", "L1", "V1"), 21, 16384.0, 2049),
    (("H1", "L1", "V1"), 4, 65536.0, 1001),    # windows of 6600 columns: several chunks, samples in turn
    (("H1", "V1"), 2, 262144.0, 257),
]


@pytest.mark.parametrize("i", range(len(SHAPES)))
def test_values_and_bins(G, oracle_lib, monkeypatch, i):
    monkeypatch.setenv("RIFT_ILE_TC", "0")
    dets, modes, fs, n_t = SHAPES[i]
    p = S.make_problem(dets, modes, fs, n_t=n_t, snr=12.0, seed=S.config_seed(6, 40 + i))
    th = S.prior_samples(2700, 50 + i)
    exp, ebins, _ = oracle_lib.lnL(p, th[:40], want_bins=True)
    rest = oracle_lib.lnL(p, th[-60:])
    with G.ILE(p, precision=G.RIFT_FP32, max_samples=2700) as s:
        for n in (1, 3, 5, 40):
            got, bins = s.eval(th[:n], want_bins=True)
            assert np.max(np.abs(got - exp[:n])) <= TOL
            assert np.max(np.abs(bins - ebins[:n])) <= TOL
        for n in (1024, 1025, 1216, 1217, 2700):   # unsorted | sorted, 4 | 8 samples a block
            got = s.eval(th[-n:])
            assert np.max(np.abs(got[-60:] - rest)) <= TOL
        full = s.eval(th)
        got, bins = s.eval(th, want_bins=True)
        assert np.array_equal(got, full)
        assert np.max(np.abs(bins[:40] - ebins)) <= TOL


@pytest.mark.parametrize("i", [1, 4, 6])
def test_distance_marginal(G, oracle_lib, monkeypatch, i):
    """The marginal and its per-bin values against the oracle; the sorted batch of 8 samples a
    block against the unsorted one of 4."""
    monkeypatch.setenv("RIFT_ILE_TC", "0")
    dets, modes, fs, n_t = SHAPES[i]
    p = S.make_problem(dets, modes, fs, n_t=n_t, snr=12.0, seed=S.config_seed(6, 60 + i))
    th = S.prior_samples(3000, 70 + i)
    exp, ebins, _ = oracle_lib.lnL(oracle_lib.Problem(p, dist_marg=True), th[:50], want_bins=True)
    with G.ILE(p, precision=G.RIFT_FP32, max_samples=3000, distance_marg=True) as s:
        full = s.eval(th)
        few, bins = s.eval(th[:50], want_bins=True)
    assert np.max(np.abs(full[:50] - exp)) <= TOL
    assert np.max(np.abs(few - exp)) <= TOL
    assert np.max(np.abs(bins - ebins)) <= TOL


def test_non_finite_sample(G, monkeypatch):
    monkeypatch.setenv("RIFT_ILE_TC", "0")
    p = S.make_problem(("H1", "L1"), 2, 4096.0, n_t=101, snr=12.0, seed=S.config_seed(6, 80))
    th = S.prior_samples(2000, 81)
    with G.ILE(p, precision=G.RIFT_FP32, max_samples=2000) as s:
        want = s.eval(th)
        for col in (0, 2, 5):
            bad = th.copy()
            bad[7, col] = np.nan
            with pytest.raises(G.RiftError) as e:
                s.eval(bad)
            assert e.value.code in (G.RIFT_ENONFINITE, G.RIFT_ERANGE)
            assert np.array_equal(s.eval(th), want)
