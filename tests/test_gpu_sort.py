"""GPU check of the sample sort at its edges: one block up to 4096 keys, radix passes over
2048-key tiles above.  The float64 mode's values do not depend on a sample's place in the
batch, so every sample of a sorted batch has exactly the value of the unsorted small batches,
whatever the order: a key lost, duplicated or misplaced by the sort shows."""
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


@pytest.mark.parametrize("dets", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
def test_every_sample_once(G, dets):
    p = S.make_problem(dets, n_modes=1, fs=4096.0, n_t=9, seed=S.config_seed(6, len(dets)), snr=10.0)
    counts = [513, 1023, 1025, 2047, 2049, 4095, 4096, 4097, 6144, 6145, 65536 + 31, 300001]
    th = S.prior_samples(counts[-1], 9)
    # pile half of the samples on one sky cell: long runs of equal keys
    th[::2, :2] = th[0, :2]
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=counts[-1]) as s:
        small = np.concatenate([s.eval(th[i:i + 512]) for i in range(0, 6656, 512)])
        full = s.eval(th)
        assert np.array_equal(full[:6656], small)
        for n in counts[:-1]:
            assert np.array_equal(s.eval(th[:n]), full[:n])


def test_stable_runs(G):
    """The same batch twice: the same float32 bits (the order of equal keys is the draw order)."""
    p = S.make_problem(("H1", "L1", "V1"), n_modes=5, fs=4096.0, n_t=101, seed=S.config_seed(6, 9), snr=10.0)
    for n in (3000, 4097, 150000):
        th = S.prior_samples(n, 10)
        with G.ILE(p, precision=G.RIFT_FP32, max_samples=n) as s:
            assert np.array_equal(s.eval(th), s.eval(th))
