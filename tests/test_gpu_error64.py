"""The float64 mode's error is no larger on the tensor cores than in the plain float64 kernel
(RIFT_ILE_TC=0): without data (Q = 0) a sample's value is minus its template term, whose error,
geometry included, is taken against long double arithmetic from the sample's coordinates.  The norm
of the errors over 4000 prior samples, whose distances weight them by less than 100 to 1, has a
sampling error of a few percent (both kernels have the same samples): 10%."""
import math

import numpy as np
import pytest

import ile_synth as S

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_11655_gb300 as G
    G.load(build_if_missing=True)
    return G


def template(p, theta):
    """kappa sum_k c^H U c + Re(c^T V c) in long double."""
    f, th = math.factorial, theta.astype(LD)
    h, d, psi = th[:, 0] - LD(p.gmst), th[:, 1], th[:, 2]
    sh, ch, sd, cd = np.sin(h), np.cos(h), np.sin(d), np.cos(d)
    ea, ed = np.stack([-sh, ch, 0 * h], 1), np.stack([-sd * ch, -sd * sh, cd], 1)
    c, s = np.cos(th[:, 4] / 2), np.sin(th[:, 4] / 2)
    Y = []
    for l, m in np.asarray(p.lm).tolist():
        root = np.sqrt(LD(2 * l + 1) / (4 * LD("3.14159265358979323846264338327950288")) *
                       f(l + m) * f(l - m) * f(l + 2) * f(l - 2))
        y = 0 * c
        for k in range(max(0, m - 2), min(l + m, l - 2) + 1):
            y = y + (-1) ** k * root / LD(f(k) * f(k - m + 2) * f(l + m - k) * f(l - k - 2)) * \
                c ** (2 * l + m - 2 - 2 * k) * s ** (2 * k - m + 2)
        Y.append((y * np.cos(m * th[:, 3]), -y * np.sin(m * th[:, 3])))
    yr, yi = (np.stack(a, 1) for a in zip(*Y))
    x, q = LD(p.d_ref) / th[:, 5], 0
    for k in range(p.n_det):
        D = p.det_tensor[k].reshape(3, 3).astype(LD)
        A = ((ea @ D) * ea).sum(1) - ((ed @ D) * ed).sum(1)
        B = ((ea @ (D + D.T)) * ed).sum(1)
        fr, fi = (x * (A * np.cos(2 * psi) - B * np.sin(2 * psi)))[:, None], (x * (A * np.sin(2 * psi) + B * np.cos(2 * psi)))[:, None]
        cr, ci = fr * yr - fi * yi, fr * yi + fi * yr
        ur, ui, vr, vi = (a.astype(LD) for a in (p.U[k].real, p.U[k].imag, p.V[k].real, p.V[k].imag))
        q = q + (cr * (cr @ ur.T - ci @ ui.T) + ci * (cr @ ui.T + ci @ ur.T)).sum(1)
        q = q + (cr * (cr @ vr.T - ci @ vi.T) - ci * (cr @ vi.T + ci @ vr.T)).sum(1)
    return q * (0.5 if p.quad_norm else 0.25)


@pytest.mark.parametrize("dets,modes", [(("H1",), 1), (("H1", "L1"), 2), (("H1", "L1", "V1"), 4), (("H1", "L1"), 9),
                                        (("L1",), 12), (("H1", "L1"), 16), (("H1", "L1", "V1"), 21)])
def test_error_of_the_template_term(G, monkeypatch, dets, modes):
    n = 4000
    p = S.make_problem(dets, modes, 4096.0, n_t=65, snr=30.0, seed=S.config_seed(6, 160 + modes))
    th = S.prior_samples(n, 161, p.d_min, p.d_max)
    want = -template(p, th)
    err = []
    for env in ("0", "2"):   # plain kernel, tensor cores
        monkeypatch.setenv("RIFT_ILE_TC", env)
        with G.ILE(p, precision=G.RIFT_FP64, max_samples=n) as s:
            s.set_overlaps(np.zeros_like(p.Q), p.U, p.V)
            err.append(float(np.linalg.norm((s.eval(th).astype(LD) - want).astype(np.float64))))
    rel = [e / float(np.linalg.norm(want.astype(np.float64))) for e in err]
    print("relative error: plain %.2e, tensor cores %.2e" % tuple(rel))
    assert rel[1] <= 1.1 * rel[0], rel
