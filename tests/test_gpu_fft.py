"""GPU check of the pruned transform behind Q at the edges of its plan: transform lengths that
are odd and even powers of two, one to 64 interleaved transforms, and the radix-2 transform
beyond; against the direct sum of the same inputs (forced by RIFT_ILE_DFT=1), to 1e-12 of
max |Q| like the other transform checks; and U, V for few and many modes against plain sums."""
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


def inputs(n_freq, df, K, M, seed):
    rng = np.random.default_rng(seed)
    fpos = (np.arange(n_freq // 2) + 0.5) * df
    f = np.concatenate([-fpos[::-1], fpos])
    h, d = ((rng.normal(size=(n, n_freq)) + 1j * rng.normal(size=(n, n_freq))) / np.sqrt(n_freq) for n in (M, K))
    wpos = rng.uniform(0.5, 2.0, size=(K, n_freq // 2))
    return f, h, d, np.concatenate([wpos[:, ::-1], wpos], axis=1)


@pytest.mark.parametrize("fs,lg,n_freq,modes", [
    (2048.0, 9, 500, 1), (2048.0, 15, 1000, 2), (2048.0, 16, 600, 2),      # P = 512: R = 1, 64, 128 (radix-2)
    (4096.0, 10, 1022, 3), (4096.0, 14, 16384, 2), (4096.0, 17, 300, 1),   # P = 1024: R = 1, 16, 128 (radix-2)
    (8192.0, 13, 8000, 5), (16384.0, 16, 700, 32),                          # P = 2048: R = 4; P = 4096: R = 16
])
def test_transform_and_template_sums(G, monkeypatch, fs, lg, n_freq, modes):
    dets = ("H1", "L1")
    lm = [(l, m) for l in range(2, 6) for m in range(-l, l + 1)][:modes]
    p = S.make_problem(dets, fs=fs, lm=lm, n_t=11, snr=10.0, seed=S.config_seed(3, 90))
    f, h, d, w = inputs(n_freq, fs / (1 << lg), len(dets), modes, lg)
    got = {}
    for dft in ("0", "1"):
        monkeypatch.setenv("RIFT_ILE_DFT", dft)
        with G.ILE(p, precision=G.RIFT_FP64, max_samples=16, set_overlaps=False) as s:
            s.set_waveforms(f, h, d, w)
            got[dft] = s.get_overlaps(p.n_q)
    (Q, U, V), (Qd, Ud, Vd) = got["0"], got["1"]
    assert np.max(np.abs(Q - Qd)) <= 1e-12 * np.max(np.abs(Qd))
    assert np.array_equal(U, Ud) and np.array_equal(V, Vd)
    Ux = np.stack([2 * (h.conj() * w[k]) @ h.T for k in range(len(dets))])
    Vx = np.stack([2 * (h[:, ::-1] * w[k]) @ h.T for k in range(len(dets))])
    assert np.max(np.abs(U - Ux)) <= 1e-13 * np.max(np.abs(Ux))
    assert np.max(np.abs(V - Vx)) <= 1e-13 * np.max(np.abs(Ux))


def test_first_violation_decides(G):
    """The error of the lowest offending frequency is reported, the grid's before the weights'."""
    p = S.make_problem(("H1", "L1"), 2, 4096.0, n_t=11, snr=10.0, seed=S.config_seed(3, 91))
    f, h, d, w = inputs(1000, 4.0, 2, 2, 1)
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=16, set_overlaps=False) as s:
        def code(ff, ww):
            with pytest.raises(G.RiftError) as e:
                s.set_waveforms(ff, h, d, ww)
            return e.value.code
        w1 = w.copy()
        w1[1, 3] = np.inf
        assert code(f, w1) == G.RIFT_ENONFINITE
        w2 = w1.copy()
        w2[0, 3] = -1.0
        assert code(f, w2) == G.RIFT_EINVAL
        f2 = f.copy()
        f2[3] = np.nan
        assert code(f2, w1) == G.RIFT_EINVAL
        f2 = f.copy()
        f2[4] = np.nan
        assert code(f2, w1) == G.RIFT_ENONFINITE
        s.set_waveforms(f, h, d, w)
