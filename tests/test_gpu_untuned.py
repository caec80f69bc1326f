"""The untuned float32 evaluation's accuracy does not depend on the batch size up to 100,000 samples:
a loud event's samples in one sorted batch carry the rounding that they carry a thousand at a time
(float32 products; float16 pairs have four times the rms error at SNR 150)."""
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


@pytest.mark.parametrize("dets,modes,fs,n_t", [(("H1", "L1", "V1"), 9, 4096.0, 403), (("L1",), 12, 16384.0, 701)])
@pytest.mark.parametrize("n", [20011, 60001])
def test_accuracy_of_larger_batches(G, monkeypatch, dets, modes, fs, n_t, n):
    monkeypatch.delenv("RIFT_ILE_TC", raising=False)
    p = S.make_problem(dets, modes, fs, n_t=n_t, snr=150.0, seed=S.config_seed(6, 150))
    th = S.prior_samples(n, 151)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
        want = s.eval(th)
    with G.ILE(p, precision=G.RIFT_FP32, max_samples=n) as s:
        whole = s.eval(th)
        parts = np.concatenate([s.eval(th[i:i + 1000]) for i in range(0, n, 1000)])
    rms = [float(np.sqrt(np.mean((x - want) ** 2))) for x in (whole, parts)]
    assert rms[0] <= 1.25 * rms[1], rms
