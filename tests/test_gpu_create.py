"""Creating a handle costs device allocations, not host arithmetic that grows with the problem: the
polar functions' tables (with the modes) and the bins' positions in fixed point (with the time grid)
are a few microseconds, where long double arithmetic, emulated on some hosts, took 1.4 ms for 21
modes and 0.1 us a bin."""
import time

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


def create_us(G, prob, precision):
    best = float("inf")
    for _ in range(30):
        t = time.perf_counter()
        h = G.ILE(prob, precision=precision, max_samples=2000, set_overlaps=False)
        best = min(best, time.perf_counter() - t)
        h.close()
    return 1e6 * best


def test_modes(G):
    few, many = (S.make_problem(("H1",), m, 4096.0, n_t=101, seed=S.config_seed(6, 120)) for m in (1, 21))
    for prec in (G.RIFT_FP32, G.RIFT_MIXED):
        a, b = create_us(G, few, prec), create_us(G, many, prec)
        assert b - a < 400.0, (a, b)   # measured 12; the buffers differ by a few megabytes


def test_time_bins(G):
    short, long = (S.make_problem(("H1",), 2, 4096.0, n_t=n, seed=S.config_seed(6, 121)) for n in (2, 3900))
    a, b = create_us(G, short, G.RIFT_FP64), create_us(G, long, G.RIFT_FP64)
    assert b - a < 200.0, (a, b)
