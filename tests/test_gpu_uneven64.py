"""Overlaps of very different sizes in the float64 mode, whose tensor-core kernel has one fixed-point
scale for Q: a large column that no bin reaches changes nothing; a detector, the modes that are
alone in a face-on sample, or a single column far above the rest take the plain float64 kernel, in
captured sequences too; overlaps of ordinary sizes stay on the tensor cores."""
import numpy as np
import pytest

import ile_synth as S

pytestmark = pytest.mark.gpu
N = 3000


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_11655_gb300 as G
    G.load(build_if_missing=True)
    return G


def problem():
    return S.make_problem(("H1", "L1", "V1"), 5, 4096.0, n_t=201, snr=20.0, seed=S.config_seed(6, 170))


def uneven(p, what):
    """Q of the problem, changed: by `what`, whether the plain kernel is due."""
    Q = p.Q.copy()
    if what == "ordinary":
        Q[2] /= 20.0
    if what == "unreachable column":   # the Q window begins 29 ms before the earliest bin
        Q[0, :, 3] = 1e9
        Q[1, 0, -2] = 1e12
    if what == "detector":
        Q[1] *= 1e5
    if what == "quiet detector":
        Q[2] /= 1e5
    if what == "face-on":
        Q[:, p.lm[:, 1] == 2] /= 1e5
    if what == "column":
        Q[0, 1, Q.shape[2] // 2] += 1e6 * np.abs(Q).max()
    if what == "silent detector":
        Q[1] = 0.0
    return Q


def values(G, monkeypatch, p, Q, env, prec=None):
    monkeypatch.setenv("RIFT_ILE_TC", env)
    th = S.prior_samples(N, 171, p.d_min, p.d_max)
    with G.ILE(p, precision=G.RIFT_FP64 if prec is None else prec, max_samples=N) as s:
        s.set_overlaps(Q, p.U, p.V)
        return s.eval(th)


@pytest.mark.parametrize("what,plain", [("ordinary", False), ("silent detector", False), ("detector", True),
                                        ("quiet detector", True), ("face-on", True), ("column", True)])
def test_kernel_by_unevenness(G, monkeypatch, what, plain):
    p = problem()
    Q = uneven(p, what)
    ref, got = (values(G, monkeypatch, p, Q, env) for env in ("0", "2"))
    assert np.array_equal(ref, got) == plain
    assert np.allclose(ref, got, rtol=1e-11, atol=1e-11)
    if plain:   # the weighted samples of the mixed mode too
        mixed = values(G, monkeypatch, p, Q, "2", G.RIFT_MIXED)
        top = ref >= ref.max() - 39.0
        assert np.allclose(mixed[top], ref[top], rtol=1e-11, atol=1e-11)


def test_unreachable_column(G, monkeypatch):
    p = problem()
    a, b = (values(G, monkeypatch, p, uneven(p, w), "2") for w in ("", "unreachable column"))
    assert np.array_equal(a, b)


def test_captured_sequences(G):
    """New overlaps on a handle whose sequence has been captured: another kernel, another capture."""
    p = problem()
    Q = uneven(p, "detector")
    with G.ILE(p, precision=G.RIFT_FP64, max_samples=N, seed=5) as s, G.ILE(p, precision=G.RIFT_FP64, max_samples=N, seed=5) as t:
        state = s.get_state()
        for _ in range(3):
            s.adapt(1, N)
        s.set_overlaps(Q, p.U, p.V)
        s.set_state(state)
        t.set_overlaps(Q, p.U, p.V)
        with G.Batch([s], [1], [N]) as batch:
            batch.run()
            first = s.last_batch(N)
            s.set_overlaps(p.Q, p.U, p.V)
            s.set_state(state)
            batch.run()
            back = s.last_batch(N)
        t.adapt(1, N)
        for x, y in zip(first, t.last_batch(N)):
            assert np.array_equal(x, y)
        t.set_overlaps(p.Q, p.U, p.V)
        t.set_state(state)
        t.adapt(1, N)
        for x, y in zip(back, t.last_batch(N)):
            assert np.array_equal(x, y)
