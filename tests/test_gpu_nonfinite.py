"""Samples with a non-finite coordinate in the float32 likelihoods: a sky angle that is not finite
has no Q index (RIFT_ERANGE, as in the float64 mode), any other coordinate no ln L
(RIFT_ENONFINITE); no address is formed from such a sample, whatever the number of time chunks, and
the handle's next evaluation is unaffected."""
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


# detectors, modes, sampling rate, time bins: one chunk of time bins, and several
SHAPES = [
    (("H1", "L1"), 2, 4096.0, 101),
    (("H1", "L1", "V1"), 5, 16384.0, 2049),
    (("H1", "L1", "V1"), 4, 65536.0, 1201),
    (("H1", "V1"), 2, 262144.0, 257),
]


@pytest.mark.parametrize("tensor", ["0", "1"])
@pytest.mark.parametrize("i", range(len(SHAPES)))
def test_non_finite_sample(G, monkeypatch, i, tensor):
    monkeypatch.setenv("RIFT_ILE_TC", tensor)
    dets, modes, fs, n_t = SHAPES[i]
    p = S.make_problem(dets, modes, fs, n_t=n_t, snr=12.0, seed=S.config_seed(6, 90 + i))
    th = S.prior_samples(2000, 91 + i)
    with G.ILE(p, precision=G.RIFT_FP32, max_samples=2000) as s:
        want = s.eval(th)
        for n in (5, 2000):   # unsorted | sorted
            for at, col, bad, code in ((0, 0, np.nan, G.RIFT_ERANGE), (n - 1, 1, np.inf, G.RIFT_ERANGE),
                                       (n // 2, 2, np.nan, G.RIFT_ENONFINITE), (0, 5, np.nan, G.RIFT_ENONFINITE)):
                x = th[:n].copy()
                x[at, col] = bad
                with pytest.raises(G.RiftError) as e:
                    s.eval(x)
                assert e.value.code == code
        x = th.copy()
        x[::3, 0] = np.nan   # whole tiles of them behind the sort
        with pytest.raises(G.RiftError) as e:
            s.eval(x)
        assert e.value.code == G.RIFT_ERANGE
        assert np.array_equal(s.eval(th), want)
