"""The handle's count of kernel launches against the profiler's list, at the sizes where a call's
kernels change (unsorted, one-block sort, radix sort, planned work units)."""
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


def seen(f):
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        f()
        torch.cuda.synchronize()
    return sum(1 for e in prof.events() if "rift::" in e.name)


@pytest.mark.parametrize("mode", ["RIFT_FP64", "RIFT_FP32", "RIFT_MIXED"])
@pytest.mark.parametrize("n", [100, 700, 5000, 20011])
def test_counts(G, mode, n):
    p = S.make_problem(("H1", "L1"), 2, 4096.0, n_t=201, snr=15.0, seed=S.config_seed(6, 130))
    th = S.prior_samples(n, 131)
    with G.ILE(p, precision=getattr(G, mode), max_samples=n) as h:
        calls = [lambda: h.eval(th), lambda: h.marginalize(n), lambda: h.adapt(2, n)]
        if n > 5000:
            calls.append(lambda: (h.marginalize(n), h.fair_draws(3000)))
        for f in calls:
            f()   # plans and attributes
        if seen(calls[0]) == 0 and seen(calls[0]) == 0:   # (the first list of a process may be empty)
            pytest.skip("no kernel activities from the profiler")
        for f in calls:
            a = G.rift_ile_kernel_launches(h.h)
            k = seen(f)
            assert G.rift_ile_kernel_launches(h.h) - a == k


@pytest.mark.parametrize("modes,cap", [(2, 64), (21, 32)])
def test_many_draws_from_a_small_handle(G, modes, cap):
    """Draws beyond a small handle's batch size are not evaluated in chunks of it, a sort and a
    tensor-core launch each; the draws are those of a large handle."""
    import numpy as np
    p = S.make_problem(("H1", "L1"), modes, 4096.0, n_t=201, snr=15.0, seed=S.config_seed(6, 132))
    out = []
    for size in (cap, 6000):
        with G.ILE(p, precision=G.RIFT_FP64, max_samples=size, seed=4) as h:
            h.marginalize(cap)
            a = G.rift_ile_kernel_launches(h.h)
            out.append(h.fair_draws(5000, seed=9))
            assert G.rift_ile_kernel_launches(h.h) - a <= 24
    for x, y in zip(*out):
        assert np.array_equal(x, y)
