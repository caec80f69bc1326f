"""What the library is timed on: the calls that a program running extrinsic-marginalised
likelihood integrals makes, through the Python binding's public names, over the sizes of
this repository's workloads (1-3 detectors, 1-21 modes, 4096 or 16384 Hz, up to 1201 time
bins, 64 to 1e6 samples).

Every problem is a seeded synthetic one of ``ile_synth`` with a physically realisable
injection.  The float32 and mixed modes return their values as float32, which is what those
modes carry (the binding's arrays are float64 whatever the mode); the float64 mode returns
float64.  ``exact`` restates the method in plain float64 torch.
"""
import math

import numpy as np
import torch

import ile_synth as S
import paper_2505_11655_gb300 as G

C_SI = 299792458.0
DETECTORS = ("H1", "L1", "V1")
PRECISIONS = {"float64": G.RIFT_FP64, "float32": G.RIFT_FP32, "mixed": G.RIFT_MIXED}
N_BINS = 64
FLOOR = 0.1

PLAIN = dict(n_det=2, n_modes=2, fs=4096.0, n_t=401, snr=20.0)
LARGE = dict(n_det=3, n_modes=21, fs=16384.0, n_t=1001, snr=20.0)


def listed():
    return [
        # a handful of parameter points looked up by another sampler: latency and launches
        dict(PLAIN, name="eval_256", kind="eval", precision="float32", n=256, bins=False, host=False),
        # a user's own set of samples, an ordinary two-detector problem, a ragged count
        dict(name="eval_30k", kind="eval", precision="float32", n=30011, bins=False, host=False, n_det=2, n_modes=9,
             fs=16384.0, n_t=1001, snr=20.0),
        # the reference precision on the largest problem
        dict(LARGE, name="eval_f64_20k", kind="eval", precision="float64", n=20011, bins=False, host=False),
        # the evidence of the largest problem with an adapted sampler (the bench's size)
        dict(LARGE, name="evidence_1m", kind="evidence", precision="float32", n=1000000, distance=False),
        # the same with the distance marginalised in every time bin
        dict(LARGE, name="evidence_distance_250k", kind="evidence", precision="float32", n=250000, distance=True),
        # a loud event: a whole adaptive solve of a new point on a kept handle, mixed precision
        dict(LARGE, name="adapt_loud_4x250k", kind="adapt", precision="mixed", n=250000, n_iter=4) | dict(snr=150.0),
        # a small request as a service takes it: handle, overlaps from the host, one iteration, samples
        dict(PLAIN, name="solve_10k", kind="solve", precision="float32", n=10000),
        # uneven points (the batched workload's sizes) as one graph
        dict(name="batch_12", kind="batch", precision="mixed", points=12, first=0, n_iter=2, shrink=3),
        # the adaptive-volume integrator, three iterations from the whole cube
        dict(name="volume_3x200k", kind="volume", precision="mixed", n=200000, n_iter=3, n_det=2, n_modes=9, fs=4096.0,
             n_t=401, snr=12.0),
        # the three-member portfolio, two iterations from its start
        dict(name="portfolio_2x200k", kind="portfolio", precision="mixed", n=200000, n_iter=2, components=4, n_det=3,
             n_modes=9, fs=4096.0, n_t=401, snr=15.0),
        # overlaps of a new intrinsic point from its waveforms (a 4 s segment at 4096 Hz)
        dict(name="waveforms_16k", kind="waveforms", precision="float64", n_freq=16384, df=0.25, n_det=3, n_modes=21,
             fs=4096.0, n_t=401, snr=20.0),
        # posterior samples with their times from a finished batch
        dict(PLAIN, name="fair_draws_4k", kind="fair", precision="float64", n=50000, n_draws=4000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    n_modes = rng.randint(1, 21)
    fs = 4096.0 if n_modes <= 4 else rng.choice([4096.0, 16384.0])
    size = dict(n_det=rng.randint(1, 3), n_modes=n_modes, fs=fs, n_t=rng.choice([401, 1001, rng.randint(101, 1201)]),
                snr=round(rng.uniform(8.0, 40.0), 2))
    kind = rng.choice(["eval", "eval", "eval", "eval64", "evidence", "evidence", "distance", "adapt", "solve",
                       "batch", "volume", "portfolio", "waveforms", "fair"])
    if kind == "eval":
        bins = rng.random() < 0.25
        return dict(size, kind="eval", precision=rng.choice(["float32", "float32", "mixed"]), bins=bins,
                    n=_log_int(rng, 64, 20000 if bins else 300000), host=rng.random() < 0.25)
    if kind == "eval64":
        return dict(size, kind="eval", precision="float64", bins=rng.random() < 0.25, n=_log_int(rng, 64, 20000),
                    host=rng.random() < 0.25)
    if kind == "evidence":
        return dict(size, kind="evidence", precision=rng.choice(["float32", "float32", "mixed"]),
                    n=_log_int(rng, 1000, 1000000), distance=False)
    if kind == "distance":
        return dict(size, kind="evidence", precision="float32", n=_log_int(rng, 1000, 250000), distance=True)
    if kind == "adapt":
        return dict(size, kind="adapt", precision="mixed", n=_log_int(rng, 3000, 250000), n_iter=rng.randint(2, 4)) | \
            dict(snr=round(rng.uniform(20.0, 150.0), 1))
    if kind == "solve":
        return dict(size, kind="solve", precision="float32", n=_log_int(rng, 3000, 100000))
    if kind == "batch":
        return dict(kind="batch", precision="mixed", points=rng.randint(4, 12), first=rng.randint(12, 480),
                    n_iter=rng.randint(1, 2), shrink=rng.randint(3, 6))
    if kind == "volume":
        return dict(size, kind="volume", precision="mixed", n=_log_int(rng, 10000, 200000), n_iter=rng.randint(1, 3))
    if kind == "portfolio":
        return dict(size, kind="portfolio", precision="mixed", n=_log_int(rng, 10000, 200000),
                    n_iter=rng.randint(1, 2), components=rng.randint(1, 8))
    if kind == "waveforms":
        lg = rng.randint(9, 14)
        return dict(size, kind="waveforms", precision="float64", n_freq=(1 << lg) - 2 * rng.randint(0, 40),
                    df=4096.0 / (1 << lg)) | dict(fs=4096.0)
    return dict(size, kind="fair", precision="float64", n=_log_int(rng, 3000, 20000), n_draws=_log_int(rng, 50, 5000)) | \
        dict(fs=4096.0)


# ------------------------------------------------------------------------------ inputs


def _problem(case, seed):
    """A seeded problem with the injection at a drawn sky position, orientation and distance,
    and that injection's prior-CDF coordinates."""
    rng = np.random.default_rng(seed)
    u = rng.uniform(0.1, 0.9, 6)
    d_true = 300.0 + 200.0 * u[5]
    gmst = float(rng.uniform(0.0, 2.0 * math.pi))
    th = np.array([[2 * math.pi * u[0], math.asin(2 * u[1] - 1), math.pi * u[2], 2 * math.pi * u[3],
                    math.acos(1 - 2 * u[4]), d_true]])
    dets = DETECTORS[:case["n_det"]]
    geo = [S.detector_geometry(d) for d in dets]
    lm = S.default_modes(case["n_modes"])
    t = torch.from_numpy(th)
    F, dt = _response(t, np.array([g[0] for g in geo]), np.array([g[1] for g in geo]), gmst)
    a0 = (F[:, :, None] * _harmonics(t, lm)[:, None, :])[0].numpy()
    prob = S.make_problem(dets, case["n_modes"], case["fs"], n_t=case["n_t"], snr=case["snr"], seed=int(seed), a0=a0,
                          dt_true=dt[0].numpy(), d_true=d_true, gmst=gmst)
    v = u.copy()
    v[5] = (d_true ** 3 - prob.d_min ** 3) / (prob.d_max ** 3 - prob.d_min ** 3)
    return prob, v


def _masses(v, seed):
    """Masses of a sampler that has adapted: a bump around the injection in every coordinate
    over the uniform floor."""
    rng = np.random.default_rng(seed + 1)
    width = np.array([0.05, 0.06, 0.25, 0.25, 0.15, 0.08]) * rng.uniform(0.7, 1.4, 6)
    x = (np.arange(N_BINS) + 0.5) / N_BINS
    bump = np.exp(-0.5 * ((x[None] - v[:, None]) / width[:, None]) ** 2)
    return (1 - FLOOR) * bump / bump.sum(1, keepdims=True) + FLOOR / N_BINS


def _handle(case, prob, seed, n, **more):
    return G.ILE(prob, precision=PRECISIONS[case["precision"]], max_samples=n, n_bins=N_BINS, adapt_floor=FLOOR,
                 seed=seed + 1, **more)


def _set_masses(h, P):
    blob = h.get_state()   # ends with the masses [6][n_bins]
    h.set_state(blob[:-P.nbytes] + np.ascontiguousarray(P).tobytes())


def _spectra(case, seed):
    """Frequency-domain inputs on a mirror-symmetric lattice."""
    rng = np.random.default_rng(seed + 2)
    K, M, F = case["n_det"], case["n_modes"], case["n_freq"]
    fpos = (np.arange(F // 2) + 0.5) * case["df"]
    f = np.concatenate([-fpos[::-1], fpos])
    h, d = ((rng.standard_normal((n, F)) + 1j * rng.standard_normal((n, F))) / math.sqrt(F) for n in (M, K))
    wpos = rng.uniform(0.5, 2.0, (K, F // 2))
    return f, h, d, np.concatenate([wpos[:, ::-1], wpos], axis=1)


def prepare(case, seed):
    kind, st = case["kind"], {"case": case, "seed": seed}
    if kind == "batch":
        solves, n = [], []
        for i in range(case["points"]):
            spec = S.batched_problem_spec(case["first"] + i)
            point = dict(n_det=len(spec["det_names"]), n_modes=spec["n_modes"], fs=spec["fs"], n_t=spec["n_t"],
                         snr=spec["snr"])
            n.append(max(2000, spec["n_samples"] // case["shrink"] // 3))
            solves.append(_handle(case, _problem(point, 100 * seed + i)[0], 100 * seed + i, n[-1]))
        return dict(st, h=solves, n=n, batch=G.Batch(solves, [case["n_iter"]] * len(n), n))
    prob, v = _problem(case, seed)
    if kind == "eval":
        theta = S.prior_samples(case["n"], seed + 3, prob.d_min, prob.d_max)
        st["theta"] = theta if case["host"] else torch.from_numpy(theta).cuda()
    if kind == "solve":
        return dict(st, prob=prob)
    if kind == "waveforms":
        st["spectra"] = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in _spectra(case, seed)]
        st["n_q"] = prob.n_q
        st["h"] = _handle(case, prob, seed, 16, set_overlaps=False)
        return st
    st["h"] = _handle(case, prob, seed, case["n"], distance_marg=bool(case.get("distance")))
    if kind in ("evidence", "fair"):
        _set_masses(st["h"], _masses(v, seed))
    if kind == "fair":
        st["h"].marginalize(case["n"])
    if kind == "adapt":
        st["fresh"] = st["h"].get_state()
    return st


# ------------------------------------------------------------------------------ the calls


def _carried(case, x):
    """Values as the case's mode carries them."""
    if case["precision"] == "float64":
        return x
    return x.float() if isinstance(x, torch.Tensor) else np.asarray(x, np.float32)


def _evidence(case, r):
    return _carried(case, np.array([r["lnZ"], r["sigma_lnZ"], r["lnL_max"]]))


def _batch(case, h, n):
    """ln L and ln w of the last batch, left on the device (the effective sample counts follow
    from ln w)."""
    out = torch.empty((2, n), dtype=torch.float64, device="cuda")
    G.rift_ile_last_batch(h.h, None, None, out[0], out[1], mem=G.RIFT_MEM_DEVICE)
    return _carried(case, out)


def run(state):
    case, h = state["case"], state.get("h")
    kind = case["kind"]
    if kind == "eval":
        if case["bins"]:
            return [_carried(case, x) for x in h.eval(state["theta"], want_bins=True)]
        return _carried(case, h.eval(state["theta"]))
    if kind == "evidence":
        r = h.marginalize(case["n"])
        return {"evidence": _evidence(case, r), "batch": _batch(case, h, case["n"])}
    if kind == "adapt":
        h.set_state(state["fresh"])
        r = h.adapt(case["n_iter"], case["n"])
        return {"evidence": _evidence(case, r), "batch": _batch(case, h, case["n"]), "masses": _carried(case, h.sampler())}
    if kind == "solve":
        with _handle(case, state["prob"], state["seed"], case["n"]) as h:
            r = h.adapt(1, case["n"])
            return {"evidence": _evidence(case, r), "batch": _batch(case, h, case["n"])}
    if kind == "batch":
        res, rc = state["batch"].run()
        if rc != 0:
            raise G.RiftError(rc, "batch")
        return {"evidence": [_evidence(case, r) for r in res],
                "batch": [_batch(case, s, n) for s, n in zip(h, state["n"])]}
    if kind == "volume":
        r = h.av(case["n_iter"], case["n"], restart=True)
        info = h.av_info()
        return {"evidence": _evidence(case, r), "batch": _batch(case, h, case["n"]),
                "cells": info["n_cells"], "live": info["n_live"], "volume": info["V"]}
    if kind == "portfolio":
        r = h.portfolio(case["n_iter"], case["n"], members=G.RIFT_MEMBER_HIST | G.RIFT_MEMBER_AV | G.RIFT_MEMBER_GMM,
                        gmm_components=case["components"], restart=True)
        pi, mu, sig = h.portfolio_gmm()
        return {"evidence": _evidence(case, r), "batch": _batch(case, h, case["n"]), "masses": _carried(case, h.sampler()),
                "mixture": [_carried(case, x) for x in (pi, mu, sig)]}
    if kind == "waveforms":
        h.set_waveforms(*state["spectra"])
        K, M = case["n_det"], case["n_modes"]
        Q, U, V = (torch.empty((K, M, n), dtype=torch.complex128, device="cuda") for n in (state["n_q"], M, M))
        G.rift_ile_get_overlaps(h.h, Q, U, V)
        return [Q, U, V]
    if kind == "fair":
        m = case["n_draws"]
        th, t = (torch.empty(s, dtype=torch.float64, device="cuda") for s in ((m, 6), (m,)))
        index = torch.empty(m, dtype=torch.int64, device="cuda")
        G.rift_ile_fair_draws(h.h, m, 7, th, t, index)
        return {"theta": th, "t": t, "index": index}
    raise ValueError(kind)


# ------------------------------------------------------------------------------ work


def _overlap_bytes(c):
    n_q = round(0.2 * c["fs"])
    return 16 * c["n_det"] * c["n_modes"] * (n_q + 2 * c["n_modes"])


def _flops(c, distance=False):
    """Of one sample's time-marginalised ln L: the mode sum on the Q grid, interpolation, template
    term, log-sum-exp (and, with the distance marginalised, one evaluation of its value a bin)."""
    K, M, nt = c["n_det"], c["n_modes"], c["n_t"]
    return K * (4 * M * (0.1 * c["fs"] + 2) + 3 * nt) + 8 * K * M * M + 3 * nt + (20 * nt if distance else 0)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for i in range(case["points"]):
            spec = S.batched_problem_spec(case["first"] + i)
            point = dict(n_det=len(spec["det_names"]), n_modes=spec["n_modes"], fs=spec["fs"], n_t=spec["n_t"])
            n = max(2000, spec["n_samples"] // case["shrink"] // 3)
            b += 16 * n + _overlap_bytes(point)
            f += case["n_iter"] * n * _flops(point)
        return {"bytes": b, "flops": f}
    if kind == "waveforms":
        K, M, F = case["n_det"], case["n_modes"], case["n_freq"]
        L = case["fs"] / case["df"]
        return {"bytes": 16 * F * (M + K) + 8 * F * (K + 1) + _overlap_bytes(case),
                "flops": K * M * 5 * L * math.log2(L) + 8 * K * M * (M + 1) * F}
    if kind == "fair":
        return {"bytes": 8 * case["n"] + 64 * case["n_draws"] + _overlap_bytes(case),
                "flops": case["n_draws"] * _flops(case)}
    n, it = case["n"], case.get("n_iter", 1)
    b = _overlap_bytes(case) + 16 * n
    if kind == "eval":
        b += 48 * n - 8 * n + (8 * n * case["n_t"] if case["bins"] else 0)
    return {"bytes": b, "flops": it * n * _flops(case, bool(case.get("distance")))}


# ------------------------------------------------------------------------------ in 64 bits


def _response(th, tensor, pos, gmst):
    """F_k [n][K] (complex) and the arrival delays [n][K]."""
    D, x = (torch.from_numpy(np.ascontiguousarray(a)).to(th) for a in (tensor, pos))
    h, d, psi = th[:, 0] - gmst, th[:, 1], th[:, 2]
    sh, ch, sd, cd = torch.sin(h), torch.cos(h), torch.sin(d), torch.cos(d)
    ea, ed = torch.stack([-sh, ch, 0 * h], 1), torch.stack([-sd * ch, -sd * sh, cd], 1)
    n = torch.stack([cd * ch, cd * sh, sd], 1)
    A, B, X = (torch.einsum("ni,kij,nj->nk", p, D, q) for p, q in ((ea, ea), (ed, ed), (ea, ed)))
    F = torch.complex(A - B, 2 * X) * torch.exp(2j * psi)[:, None]
    return F, -(n @ x.T) / C_SI


def _harmonics(th, lm):
    """-2Y_lm(iota, -phi) [n][M], from the closed sum of the Wigner small-d."""
    f = math.factorial
    c, s = torch.cos(0.5 * th[:, 4]), torch.sin(0.5 * th[:, 4])
    out = []
    for l, m in np.asarray(lm).tolist():
        root = math.sqrt((2 * l + 1) / (4 * math.pi) * f(l + m) * f(l - m) * f(l + 2) * f(l - 2))
        d = 0 * c
        for k in range(max(0, m - 2), min(l + m, l - 2) + 1):
            d = d + (-1) ** k * root / (f(k) * f(k - m + 2) * f(l + m - k) * f(l - k - 2)) * \
                c ** (2 * l + m - 2 - 2 * k) * s ** (2 * k - m + 2)
        out.append(d * torch.exp(-1j * m * th[:, 3]))
    return torch.stack(out, 1)


def _ln_distance(prob, a, b):
    """ln of the distance marginal of every bin: composite Gauss-Legendre in ln x over the part
    of the range where the exponent a x - b x^2 is within 60 of its maximum."""
    xlo, xhi = prob.d_ref / prob.d_max, prob.d_ref / prob.d_min
    xm = (a / (2 * b)).clamp(xlo, xhi)
    g = (a - 2 * b * xm).abs()
    d = 120.0 / (g + torch.sqrt(g * g + 240.0 * b))
    u0, u1 = torch.log((xm - d).clamp_min(xlo)), torch.log((xm + d).clamp_max(xhi))
    top = a * xm - b * xm * xm
    t, w = np.polynomial.legendre.leggauss(20)
    panels, total = 4, torch.zeros_like(a)
    for p in range(panels):
        for ti, wi in zip(t, w):
            u = u0 + (u1 - u0) * ((p + 0.5 * (1 + ti)) / panels)
            x = torch.exp(u)
            total += wi * torch.exp(a * x - b * x * x - top - 3 * u)
    ln_c = math.log(3 * prob.d_ref ** 3 / (prob.d_max ** 3 - prob.d_min ** 3))
    return ln_c + top + torch.log(total * (u1 - u0) / (2 * panels))


def _ln_like(prob, theta, distance=False, bins=False):
    n, K, M = theta.shape[0], prob.n_det, prob.n_modes
    dev = theta.device
    Q, U, V = (torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (prob.Q, prob.U, prob.V))
    t = torch.from_numpy(prob.t_lo + np.arange(prob.n_t) * ((prob.t_hi - prob.t_lo) / max(1, prob.n_t - 1))).to(dev)
    kappa = 0.5 if prob.quad_norm else 0.25
    out = torch.empty(n, dtype=torch.float64, device=dev)
    rows = torch.empty((n, prob.n_t), dtype=torch.float64, device=dev) if bins else None
    step = max(1, (1 << 24) // max(prob.n_q, prob.n_t))
    for i in range(0, n, step):
        th = theta[i:i + step]
        F, dt = _response(th, prob.det_tensor, prob.det_pos, prob.gmst)
        Y = _harmonics(th, prob.lm)
        x = torch.ones_like(th[:, 5]) if distance else prob.d_ref / th[:, 5]
        quad, lin = 0.0, 0.0
        for k in range(K):
            c = (x * F[:, k])[:, None] * Y
            quad = quad + kappa * ((c.conj() @ U[k] * c).sum(1).real + (c @ V[k] * c).sum(1).real)
            R = c.real.contiguous() @ Q[k].real.contiguous() + c.imag.contiguous() @ Q[k].imag.contiguous()
            u = (t[None] + (dt[:, k] - float(prob.q_t0[k]))[:, None]) * prob.fs
            lo = u.floor()
            j = lo.long()
            lin = lin + (1 - (u - lo)) * R.gather(1, j) + (u - lo) * R.gather(1, j + 1)
        lnL = _ln_distance(prob, lin, quad[:, None].expand_as(lin)) if distance else lin - quad[:, None]
        if bins:
            rows[i:i + step] = lnL
        out[i:i + step] = torch.logsumexp(lnL, 1) - math.log(prob.n_t)
    return out, rows


def _philox(i, iteration, word, seed):
    """Philox4x32-10 (Salmon et al. 2011): four 32-bit words per counter (i, iteration, word)."""
    m32 = 0xFFFFFFFF
    c = [i & m32, i >> 32, torch.full_like(i, iteration), torch.full_like(i, word)]
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        p, q = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((q >> 32) & m32) ^ c[1] ^ k0, q & m32, ((p >> 32) & m32) ^ c[3] ^ k1, p & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _draws(prob, P, n, seed, iteration, distance):
    """The product-form sampler's draws: theta, ln p - ln p_s, histogram bins."""
    i = torch.arange(n, device="cuda")
    v, lr, bins = [], torch.zeros(n, dtype=torch.float64, device="cuda"), []
    P = torch.from_numpy(np.ascontiguousarray(P)).cuda()
    words = [_philox(i, iteration, p, seed) for p in range(3)]
    for d in range(6):
        a, b = words[d // 2][2 * (d % 2):2 * (d % 2) + 2]
        u = (((a >> 5) << 26) | (b >> 6)).double() * 2.0 ** -53
        C = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), P[d].cumsum(0)])
        x = u * C[-1]
        j = (torch.searchsorted(C, x, right=True) - 1).clamp(0, N_BINS - 1)
        v.append((j + ((x - C[j]) / P[d][j]).clamp(0.0, 1.0)) / N_BINS)
        bins.append(j)
        if not (distance and d == 5):
            lr -= torch.log(N_BINS * P[d] / C[-1])[j]
    lo, hi = prob.d_min ** 3, prob.d_max ** 3
    th = torch.stack([2 * math.pi * v[0], torch.asin(2 * v[1] - 1), math.pi * v[2], 2 * math.pi * v[3],
                      torch.acos(1 - 2 * v[4]), (lo + v[5] * (hi - lo)) ** (1 / 3)], 1)
    return th, lr, bins


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        prob, _ = _problem(case, seed)
        theta = torch.from_numpy(S.prior_samples(case["n"], seed + 3, prob.d_min, prob.d_max)).cuda()
        lnL, rows = _ln_like(prob, theta, bins=case["bins"])
        return [lnL, rows] if case["bins"] else lnL
    if kind == "waveforms":
        prob, _ = _problem(case, seed)
        f, h, d, w = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in _spectra(case, seed))
        Q = []
        for k in range(case["n_det"]):
            t = float(prob.q_t0[k]) + torch.arange(prob.n_q, device="cuda").double() / prob.fs
            A = 2 * w[k] * h.conj() * d[k]
            Q.append(torch.cat([A @ torch.exp(2j * math.pi * torch.outer(f, s)) for s in t.split(256)], 1))
        U = [2 * (h.conj() * w[k]) @ h.T for k in range(case["n_det"])]
        V = [2 * (h.flip(1) * w[k]) @ h.T for k in range(case["n_det"])]
        return [torch.stack(x) for x in (Q, U, V)]
    if kind == "evidence" or kind == "solve" or (kind == "adapt" and case["n_iter"] <= 4):
        distance = bool(case.get("distance"))
        prob, v = _problem(case, seed)
        P = _masses(v, seed) if kind == "evidence" else np.full((6, N_BINS), 1.0 / N_BINS)
        lnws, lnLmax = [], []
        for it in range(case.get("n_iter", 1)):
            th, lr, bins = _draws(prob, P, case["n"], seed + 1, it, distance)
            lnL, _ = _ln_like(prob, th, distance)
            lnw = lnL + lr
            lnws.append(lnw)
            lnLmax.append(lnL.max())
            if kind == "adapt":
                w = torch.exp(lnw - lnw.max())
                H = torch.stack([torch.zeros(N_BINS, dtype=torch.float64, device="cuda").index_add_(0, j, w) for j in bins])
                P = ((1 - FLOOR) * H / H.sum(1, keepdim=True) + FLOOR / N_BINS).cpu().numpy()
        every = torch.cat(lnws)
        lnZ = torch.logsumexp(every, 0) - math.log(every.numel())
        var = torch.exp(torch.logsumexp(2 * every, 0) - 2 * torch.logsumexp(every, 0)) - 1 / every.numel()
        out = {"evidence": torch.stack([lnZ, var.clamp_min(0).sqrt(), torch.stack(lnLmax).max()]),
               "batch": torch.stack([lnL, lnw])}
        if kind == "adapt":
            out["masses"] = P
        return out
    return None
