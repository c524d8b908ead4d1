"""The work this library is used for, as cases that can be timed and checked.

Each case is one call (or one short chain of calls) of the public binding
`paper_2005_03060_gb300.gridcorr`, at sizes of the repository's own tests and
benchmark.  `listed()` names them, `draw(rng)` gives further ones of the same
ranges, `prepare` makes the inputs on the GPU, `run` does one pass, `work`
states the bytes and operations a pass cannot do without, and `exact` gives the
results in 64-bit arithmetic by plain torch, without the library's code.

Inputs follow the recipe of the repository's synthetic draws: point sources with
dN/dS ~ S^-2 seen by every antenna, receiver noise at a power SNR of 10, gains
(1 + N(0, 0.05)) exp(i U(-pi, pi)); visibility-level draws for the calibration
alone (random amplitude and phase per baseline-type, radiometer noise).
"""
from __future__ import annotations

import math

import torch

from paper_2005_03060_gb300 import gridcorr, synth

DEV = "cuda"
CHUNK = 1 << 28        # voltage elements drawn at a time
BYTES = {"c64": 8, "c32h": 4, "i4c": 1}


def listed():
    return [
        # The FFT-correlator of the benchmark's headline array (64x64 antennas, 4+4-bit voltages,
        # 8192 samples): a quarter of its 1024 channels.
        {"name": "correlate_i4c_64", "kind": "correlate", "fmt": "i4c", "L": 64, "C": 256, "T": 8192},
        # The same step on the paper-scale array in floating point.
        {"name": "correlate_c64_32", "kind": "correlate", "fmt": "c64", "L": 32, "C": 256, "T": 4096},
        # The paper's 331-antenna hexagon (a partly occupied 21 x 21 grid), binary16 voltages, a ragged
        # number of samples.
        {"name": "correlate_hex331_c32h", "kind": "correlate", "fmt": "c32h", "L": 21, "C": 128, "T": 2047, "hex": 11},
        # The largest grid the correlator takes (128x128, 256x256 FFT).
        {"name": "correlate_i4c_128", "kind": "correlate", "fmt": "i4c", "L": 128, "C": 48, "T": 1100},
        # Calibrator step (a) of the headline array: exact integer sums of the subset selection's pairs.
        {"name": "reduce_i4c_64", "kind": "reduce", "fmt": "i4c", "scheme": "subset", "L": 64, "C": 256, "T": 8192},
        # Low-cadence selection (every pair, each in its own short window), paper-scale array, complex64.
        {"name": "reduce_lowcad_c64_32", "kind": "reduce", "fmt": "c64", "scheme": "lowcad", "L": 32, "C": 64, "T": 4096},
        # calibrate() as it is called with no options (Gauss-Newton, FP64 normal equations), paper-scale array.
        {"name": "calibrate_lincal_32", "kind": "calibrate", "fmt": "c64", "scheme": "subset", "solver": "lincal",
         "L": 32, "C": 128, "T": 4096},
        # Calibrator step (b) of the headline array: the matrix-free solver on integer sums.
        {"name": "calibrate_cg_64", "kind": "calibrate", "fmt": "i4c", "scheme": "subset", "solver": "lincal_cg",
         "L": 64, "C": 512, "T": 8192},
        # Low-cadence calibration: every pair of a 24x24 array (1151 baseline-types).
        {"name": "calibrate_lowcad_24", "kind": "calibrate", "fmt": "c64", "scheme": "lowcad", "solver": "lincal_cg",
         "L": 24, "C": 64, "T": 4096},
        # The differentiable objective on the 128x128 array: chi^2 per channel and its gradients by autograd.
        {"name": "chi2_grad_128", "kind": "chi2", "fmt": "i4c", "L": 128, "C": 256, "T": 2048, "checkpoint": False},
        # The whole cycle on the smallest array of the tests, where launches and latency count.
        {"name": "cycle_c64_8", "kind": "cycle", "fmt": "c64", "L": 8, "C": 32, "T": 256},
        # The whole cycle of the paper-scale array from floating-point voltages through the quantiser.
        {"name": "cycle_i4c_32", "kind": "cycle", "fmt": "i4c", "L": 32, "C": 64, "T": 2048},
    ]


def _log(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _fit(rng, L, C, T, most, least_t):
    """C and T brought under `most` antenna-samples."""
    while C * T * L * L > most and C > 1:
        C = max(1, C // 2 + rng.randint(0, 1) if C > 2 else 1)
    while C * T * L * L > most and T > least_t:
        T = max(least_t, T // 2 + rng.randint(0, 1))
    return C, T


def draw(rng):
    kind = rng.choice(["correlate", "correlate", "reduce", "reduce", "calibrate", "calibrate", "chi2", "cycle"])
    if kind == "correlate":
        fmt = rng.choice(["c64", "c32h", "i4c", "i4c"])
        most = {"c64": 1 << 29, "c32h": 1 << 29, "i4c": 1 << 32}[fmt]
        if rng.random() < 0.2:
            s = rng.randint(3, 11)
            L, more = 2 * s - 1, {"hex": s}
            most = 1 << 28
        else:
            L, more = _log(rng, 4, 128 if fmt == "i4c" else 64), {}
            if L > 64 or (fmt == "i4c" and L not in (40, 48, 56, 64)):
                most = 1 << 29
        C, T = _fit(rng, L, _log(rng, 1, 512), _log(rng, 48, 8192), most, 48)
        return {"kind": kind, "fmt": fmt, "L": L, "C": C, "T": T, **more}
    if kind == "reduce":
        fmt = rng.choice(["c64", "c32h", "i4c", "i4c"])
        scheme = rng.choice(["subset", "subset", "lowcad"])
        L = _log(rng, 4, 96) if scheme == "subset" else _log(rng, 4, 32)
        if fmt == "i4c" and scheme == "subset" and rng.random() < 0.5:
            L = rng.choice([16, 32, 64])
        most = 1 << 28 if scheme == "lowcad" else (1 << 32 if fmt == "i4c" and L in (16, 32, 64) else 1 << 29)
        C, T = _fit(rng, L, _log(rng, 1, 512), _log(rng, 256, 8192), most, 256)
        return {"kind": kind, "fmt": fmt, "scheme": scheme, "L": L, "C": C, "T": T}
    if kind == "calibrate":
        fmt = rng.choice(["c64", "i4c"])
        solver = rng.choice(["lincal", "lincal_cg", "lincal_cg", "omnical"])
        scheme = "subset" if solver == "lincal" else rng.choice(["subset", "lowcad"])
        if solver == "lincal":
            L, C = _log(rng, 4, 32), _log(rng, 1, 128)
        elif solver == "omnical":
            L, C = _log(rng, 4, 16), _log(rng, 1, 128)
        elif scheme == "lowcad":
            L, C = _log(rng, 4, 24), _log(rng, 1, 64)
        else:
            L, C = _log(rng, 4, 64), _log(rng, 1, 512)
        return {"kind": kind, "fmt": fmt, "scheme": scheme, "solver": solver, "L": L, "C": C, "T": 1024 * rng.randint(2, 8)}
    if kind == "chi2":
        return {"kind": kind, "fmt": rng.choice(["c64", "i4c"]), "L": _log(rng, 6, 128), "C": _log(rng, 4, 256), "T": 2048,
                "checkpoint": rng.random() < 0.5}
    L = _log(rng, 6, 40)
    C, T = _fit(rng, L, _log(rng, 4, 128), _log(rng, 256, 4096), 1 << 27, 256)
    fmt = rng.choice(["c64", "i4c"])
    if fmt == "i4c":
        T += T % 2  # the quantiser takes an even number of values per channel
    return {"kind": kind, "fmt": fmt, "L": L, "C": C, "T": T}


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + stream * 104_729 + 17) & 0x7FFF_FFFF_FFFF_FFFF)
    return g


def _gains(seed, C, N):
    g = _gen(seed, 1)
    amp = 1.0 + 0.05 * torch.randn(C, N, generator=g, device=DEV, dtype=torch.float64)
    ph = (2.0 * torch.rand(C, N, generator=g, device=DEV, dtype=torch.float64) - 1.0) * math.pi
    return torch.polar(amp, ph).to(torch.complex64)


def _cnormal(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV) * math.sqrt(0.5))


def _quantised(x):
    """4+4-bit bytes of [c, T, N] voltages, one scale per channel (RMS of 3 levels per component), and the scales."""
    r = torch.view_as_real(x)
    rms = torch.stack([torch.sqrt(v.double().square().sum() / v.numel()) for v in r])
    scale = (3.0 / rms).float()
    q = r * scale.view(-1, 1, 1, 1)
    q = torch.sign(q) * torch.floor(q.abs() + 0.5)
    q = q.clamp_(-7, 7).to(torch.int16)
    return ((q[..., 0] << 4) | (q[..., 1] & 15)).to(torch.uint8), scale


def _voltages(seed, fmt, L, C, T, gains, lattice="square"):
    """[C, T, N] voltages of 20 point sources and noise, in the format asked for."""
    N, K = L * L, 20
    sky = synth.make_sky(seed, K)
    pos = synth.lattice_positions(L, lattice)
    steer = torch.polar(torch.ones((), dtype=torch.float64), 2.0 * math.pi * (sky.l @ pos.T)).to(torch.complex64).to(DEV)
    amp = sky.flux.float().sqrt().to(DEV)
    sigma = math.sqrt(float(sky.flux.sum()) / 10.0)
    out = {"c64": lambda: torch.empty(C, T, N, dtype=torch.complex64, device=DEV),
           "c32h": lambda: torch.empty(C, T, N, 2, dtype=torch.float16, device=DEV),
           "i4c": lambda: torch.empty(C, T, N, dtype=torch.uint8, device=DEV)}[fmt]()
    g = _gen(seed, 2)
    step = max(1, CHUNK // (T * N))
    for c in range(0, C, step):
        n = min(step, C - c)
        x = (_cnormal(g, n * T, K) * amp) @ steer
        x = x.view(n, T, N).add_(_cnormal(g, n, T, N), alpha=sigma).mul_(gains[c:c + n].unsqueeze(1))
        out[c:c + n] = x if fmt == "c64" else torch.view_as_real(x).half() if fmt == "c32h" else _quantised(x)[0]
    return out


def _visibilities(seed, fmt, sel, C):
    """(sums, autos, gains, V): the reduced X-engine's output for random visibilities per type, radiometer noise (SNR ~ 10)."""
    N, dev = sel.L * sel.L, DEV
    gains = _gains(seed, C, N)
    g = _gen(seed, 3)
    pi, pj, pt, tp = _pairs(sel)
    amp = 0.5 + torch.rand(C, sel.n_ubl, generator=g, device=dev, dtype=torch.float64)
    ph = (2.0 * torch.rand(C, sel.n_ubl, generator=g, device=dev, dtype=torch.float64) - 1.0) * math.pi
    V = torch.polar(amp, ph)
    power = 0.1 * math.sqrt(float(tp.max()))            # autocorrelation per unit gain: SNR 10 for the longest window
    unit = 18.0 / power if fmt == "i4c" else 1.0        # 4+4-bit voltages have a mean power of 18 levels^2
    sums = torch.empty(C, sel.P, dtype=torch.complex64, device=dev)
    for c in range(C):
        gc = gains[c].to(torch.complex128)
        noise = torch.view_as_complex(torch.randn(sel.P, 2, generator=g, device=dev, dtype=torch.float64) * math.sqrt(0.5))
        sums[c] = (unit * (gc[pi] * gc[pj].conj() * V[c][pt] * tp + gc[pi].abs() * gc[pj].abs() * power * tp.sqrt() * noise)).to(torch.complex64)
    autos = unit * power * gains.abs().double().square() * (sel.n_cycle * sel.t_int if sel.scheme == "lowcad" else sel.T)
    if fmt == "i4c":
        return torch.view_as_real(sums).round().to(torch.int32), autos.round().to(torch.int32), gains, V * unit
    return sums, autos.float(), gains, V * unit


def _pairs(sel):
    """Index tensors of the selection's pairs: i, j, type, window length."""
    t = lambda a: torch.as_tensor(a, dtype=torch.long, device=DEV)  # noqa: E731
    pt = t(sel.pair_type())
    return t(sel.pair_i), t(sel.pair_j), pt, (t(sel.win_t1) - t(sel.win_t0))[pt].double()


def prepare(case, seed):
    kind, fmt, L, C, T = (case[k] for k in ("kind", "fmt", "L", "C", "T"))
    s = {"case": dict(case), "ctx": gridcorr.default_context()}
    if kind == "correlate":
        s["gains"] = _gains(seed, C, L * L)
        s["mask"] = synth.hex_mask(case["hex"])[1] if "hex" in case else None
        s["volt"] = _voltages(seed, fmt, L, C, T, s["gains"], "triangular" if "hex" in case else "square")
    elif kind == "reduce":
        s["sel"] = gridcorr.Selection(case["scheme"], L, T)
        s["volt"] = _voltages(seed, fmt, L, C, T, _gains(seed, C, L * L))
    elif kind == "calibrate":
        s["sel"] = gridcorr.Selection(case["scheme"], L, T)
        s["vred"], s["autos"], s["truth"], s["vtruth"] = _visibilities(seed, fmt, s["sel"], C)
    elif kind == "chi2":
        s["sel"] = gridcorr.Selection("subset", L, T)
        s["vred"], _, gains, V = _visibilities(seed, fmt, s["sel"], C)
        g = _gen(seed, 4)  # a point near the minimum, as in the middle of a gradient descent
        s["gains"] = (gains * (1 + 0.02 * _cnormal(g, *gains.shape))).requires_grad_()
        s["vmodel"] = (V.to(torch.complex64) * (1 + 0.02 * _cnormal(g, *V.shape))).requires_grad_()
    else:
        s["sel"] = gridcorr.Selection("subset", L, T)
        truth = _gains(seed, C, L * L)
        s["volt"] = _voltages(seed, "c64", L, C, T, truth)
        s["gains"] = truth * (1 + 0.02 * _cnormal(_gen(seed, 4), C, L * L))  # the previous integration's
    return s


# ------------------------------------------------------------------ one pass

def _solution(gains, vmodel, stats):
    """The solver's results: gains, model, chi^2 and reduced chi^2, DoF and status per channel (views of the 32-byte
    records; the iteration counts in them say how the solver got there and are not results)."""
    return {"gains": gains, "vmodel": vmodel, "chi2": stats.view(torch.float64)[:, :2], "state": stats.view(torch.int32)[:, 4::2]}


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "correlate":
        return ctx.correlate(state["volt"], state["gains"], mask=state["mask"])
    if case["kind"] == "reduce":
        return ctx.reduce(state["volt"], state["sel"])
    if case["kind"] == "calibrate":
        return _solution(*ctx.calibrate(state["vred"], state["sel"], state["autos"], solver=case["solver"]))
    if case["kind"] == "chi2":
        gains, vmodel = state["gains"], state["vmodel"]
        chi2 = gridcorr.chi2(gains, vmodel, state["vred"], state["sel"], ctx, checkpoint=case["checkpoint"])
        return (chi2.detach(), *torch.autograd.grad(chi2.sum(), (gains, vmodel)))
    volt, more = state["volt"], {}
    if case["fmt"] == "i4c":
        volt, scales = ctx.quantize(volt)
        more = {"volt": volt, "scales": scales}
    vunique = ctx.correlate(volt, state["gains"])
    vred, autos = ctx.reduce(volt, state["sel"])
    cal = ctx.calibrate(vred, state["sel"], autos, solver="lincal_cg")
    return {"vunique": vunique, "vred": vred, "autos": autos, **_solution(*cal), **more}


# ------------------------------------------------------------------ what a pass cannot do without

def _correlate_work(case):
    L, C, T = case["L"], case["C"], case["T"]
    M = 16
    while M < 2 * L - 1:
        M *= 2
    m = math.log2(M)
    a_sample = 10 * (L * (M / 2) * (m - 1) + M * (M / 2) * m) + 4 * M * M + 6 * L * L
    return (BYTES[case["fmt"]] * C * T * L * L + 8 * C * (L * L + (2 * L - 1) ** 2), a_sample * C * T)


def _reduce_work(case, scheme):
    L, C, T = case["L"], case["C"], case["T"]
    sel = gridcorr.Selection(scheme, L, T)
    samples = float(((sel.win_t1 - sel.win_t0) * (sel.type_ptr[1:] - sel.type_ptr[:-1])).sum())
    return (BYTES[case["fmt"]] * C * T * L * L + 8 * C * sel.P + 4 * C * L * L, 8.0 * C * samples + 4.0 * C * T * L * L)


def _calibrate_work(case, scheme):
    """The sums read once, and five Gauss-Newton iterations' products per pair."""
    L, C = case["L"], case["C"]
    sel = gridcorr.Selection(scheme, L, case["T"])
    return 8 * C * sel.P + 12 * C * L * L + 8 * C * sel.n_ubl + 32 * C, 5 * 60.0 * C * sel.P


def work(case):
    kind, L, C = case["kind"], case["L"], case["C"]
    if kind == "correlate":
        b, f = _correlate_work(case)
    elif kind == "reduce":
        b, f = _reduce_work(case, case["scheme"])
    elif kind == "calibrate":
        b, f = _calibrate_work(case, case["scheme"])
    elif kind == "chi2":  # the sums once forward and once backward (the residuals, where they are kept, written and read instead)
        sel = gridcorr.Selection("subset", L, case["T"])
        b = 8 * C * sel.P * (3 if case["checkpoint"] else 2) + (2 + 1) * 8 * C * (L * L + sel.n_ubl)
        f = (20 + 50) * float(C * sel.P)
    else:
        parts = [_correlate_work(case), _reduce_work(case, "subset"), _calibrate_work(case, "subset")]
        b, f = (sum(p[k] for p in parts) for k in (0, 1))
        if case["fmt"] == "i4c":
            b += 9 * C * case["T"] * L * L
            f += 8.0 * C * case["T"] * L * L
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the results in 64 bits

def _decoded(volt):
    """complex128 voltages of any format."""
    if volt.dtype == torch.uint8:
        q = volt.to(torch.int16)
        re, im = ((q >> 4) ^ 8) - 8, ((q & 15) ^ 8) - 8
        return torch.complex(re.double(), im.double())
    return torch.view_as_complex(volt.double()) if volt.dtype == torch.float16 else volt.to(torch.complex128)


def _exact_correlate(volt, gains, L, mask):
    C, T, N = volt.shape[0], volt.shape[1], L * L
    M = 2 * L
    W = 2 * L - 1
    m = torch.ones(N, device=DEV, dtype=torch.float64) if mask is None else torch.as_tensor(mask, device=DEV).double()
    inv = torch.where(m > 0, 1.0 / gains.to(torch.complex128), 0.0)
    lags = torch.arange(-(L - 1), L, device=DEV) % M
    corr = lambda p: torch.fft.ifft2(p)[..., lags, :][..., lags]  # noqa: E731
    n_d = corr(torch.fft.fft2(m.view(L, L).to(torch.complex128), s=(M, M)).abs().square()).real.round()
    out = torch.empty(C, W, W, dtype=torch.complex128, device=DEV)
    step = max(1, (1 << 27) // (M * M))
    for c in range(C):
        p = torch.zeros(M, M, dtype=torch.float64, device=DEV)
        for t in range(0, T, step):
            x = torch.fft.fft2((_decoded(volt[c, t:t + step]) * inv[c]).view(-1, L, L), s=(M, M))
            p += torch.view_as_real(x).square_().sum(dim=(0, 3))
        out[c] = torch.where(n_d > 0, corr(p) / (T * n_d.clamp(min=1)), 0.0)
    return out


def _exact_reduce(volt, sel):
    C, T, N = volt.shape[:3]
    pi, pj, _, _ = _pairs(sel)
    used = sel.n_cycle * sel.t_int if sel.scheme == "lowcad" else sel.T
    sums = torch.empty(C, sel.P, dtype=torch.complex128, device=DEV)
    autos = torch.empty(C, N, dtype=torch.float64, device=DEV)
    many = max(1, (1 << 28) // (T * N))
    for c in range(0, C, many):
        v = _decoded(volt[c:c + many])
        autos[c:c + many] = torch.view_as_real(v[:, :used]).square().sum(dim=(1, 3))
        for k in range(sel.n_ubl):
            p = slice(int(sel.type_ptr[k]), int(sel.type_ptr[k + 1]))
            w = v[:, int(sel.win_t0[k]):int(sel.win_t1[k])]
            sums[c:c + many, p] = torch.einsum("ctp,ctp->cp", w[..., pi[p]], w[..., pj[p]].conj())
    return sums, autos


def _exact_calibrate(vred, autos, sel, gains, V):
    """The least-squares solution near (gains, V) by Gauss-Newton with dense normal equations, in the library's output
    convention: mean ln|g| = 0, arg g_0 = 0, arg V_(1,0) = arg V_(0,1) = 0."""
    L, N, K = sel.L, sel.L * sel.L, sel.n_ubl
    pi, pj, pt, tp = _pairs(sel)
    S = torch.view_as_complex(vred.double()) if vred.dtype == torch.int32 else vred.to(torch.complex128)
    obs = S / tp
    pos = synth.grid_positions(L, DEV)
    d = torch.as_tensor(sel.types, device=DEV).double()
    n = 2 * (N + K)
    G, W = gains.to(torch.complex128).clone(), V.clone()
    at = torch.stack([2 * pi, 2 * pi + 1, 2 * pj, 2 * pj + 1, 2 * (N + pt), 2 * (N + pt) + 1], 1)  # [P, 6]
    flat = (at.unsqueeze(2) * n + at.unsqueeze(1)).reshape(-1)
    for c in range(G.shape[0]):
        g, w = G[c], W[c]
        for _ in range(12):
            gi, gj, v = g[pi], g[pj].conj(), w[pt]
            J = torch.stack([gj * v, 1j * gj * v, gi * v, -1j * gi * v, gi * gj, 1j * gi * gj], 1)  # d model / d unknown
            J = torch.view_as_real(J)                                                              # [P, 6, 2]
            r = torch.view_as_real(obs[c] - gi * gj * v)
            A = torch.zeros(n * n, dtype=torch.float64, device=DEV).index_add_(0, flat, torch.einsum("pac,pbc->pab", J, J).reshape(-1)).view(n, n)
            b = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, at.reshape(-1), torch.einsum("pac,pc->pa", J, r).reshape(-1))
            z = [torch.cat([g, -2 * w]), torch.cat([1j * g, 0 * w])] + [torch.cat([1j * pos[:, a] * g, -1j * d[:, a] * w]) for a in (0, 1)]
            Z = torch.linalg.qr(torch.stack([torch.view_as_real(q).reshape(-1) for q in z], 1))[0]
            A += A.diagonal().mean() * (Z @ Z.T)
            x = torch.cholesky_solve(b.unsqueeze(1), torch.linalg.cholesky(A)).view(-1, 2)
            x = torch.view_as_complex(x)
            g, w = g + x[:N], w + x[N:]
            if float(x.abs().max()) < 1e-12 * float(w.abs().max()):
                break
        a = g.abs().log().mean().exp()
        g, w = g / a, w * a * a
        ax = [int(((d[:, 0] == e[0]) & (d[:, 1] == e[1])).nonzero()[0, 0]) for e in ((1, 0), (0, 1))]
        k = torch.stack([w[q].angle() for q in ax])
        g, w = g * torch.polar(torch.ones_like(pos[:, 0]), pos @ k), w * torch.polar(torch.ones_like(d[:, 0]), -(d @ k))
        G[c], W[c] = g * (g[0].conj() / g[0].abs()), w
    model = G[:, pi] * G[:, pj].conj() * W[:, pt]
    r2 = (obs - model).abs().square()
    used = sel.n_cycle * sel.t_int if sel.scheme == "lowcad" else sel.T
    A = autos.double() / used
    dof = sel.P - N - K + 2
    chi2 = torch.stack([r2.sum(1), (r2 / (A[:, pi] * A[:, pj] / tp)).sum(1) / dof], 1)
    return {"gains": G, "vmodel": W, "chi2": chi2, "state": None}


def _exact_chi2(s):
    sel, N = s["sel"], s["sel"].L ** 2
    pi, pj, pt, tp = _pairs(sel)
    vred = s["vred"]
    G, W = s["gains"].detach().to(torch.complex128), s["vmodel"].detach().to(torch.complex128)
    out = [], [], []
    for c in range(G.shape[0]):
        S = torch.view_as_complex(vred[c].double()) if vred.dtype == torch.int32 else vred[c].to(torch.complex128)
        g, w = G[c], W[c]
        gi, gj, v = g[pi], g[pj].conj(), w[pt]
        r = S / tp - gi * gj * v
        dg = torch.zeros(N, dtype=torch.complex128, device=DEV)
        dg.index_add_(0, pi, -2 * r * (gj * v).conj()).index_add_(0, pj, -2 * r.conj() * gi * v)
        dv = torch.zeros(sel.n_ubl, dtype=torch.complex128, device=DEV).index_add_(0, pt, -2 * r * (gi * gj).conj())
        for o, x in zip(out, (r.abs().square().sum(), dg, dv)):
            o.append(x)
    return tuple(torch.stack(o) for o in out)


def exact(case, seed):
    kind, L = case["kind"], case["L"]
    solves = 6.0 * case["C"] * (2.0 * L * L) ** 3 / 3 * 2   # flops of the dense Gauss-Newton solutions
    if kind == "calibrate" and solves > 5e12:
        return None
    if kind == "reduce" and case["fmt"] == "i4c":
        return None  # whole numbers
    s = prepare(case, seed)
    if kind == "correlate":
        return _exact_correlate(s["volt"], s["gains"], L, s["mask"])
    if kind == "reduce":
        return _exact_reduce(s["volt"], s["sel"])
    if kind == "calibrate":
        return _exact_calibrate(s["vred"], s["autos"], s["sel"], s["truth"], s["vtruth"])
    if kind == "chi2":
        return _exact_chi2(s)
    volt, more = s["volt"], {}
    if case["fmt"] == "i4c":
        volt, scales = _quantised(volt)
        more = {"scales": scales.double(), "volt": None}
    sums, autos = _exact_reduce(volt, s["sel"])
    out = {"vunique": _exact_correlate(volt, s["gains"], L, None), "vred": sums, "autos": autos, **more}
    if case["fmt"] == "i4c":
        out["vred"] = out["autos"] = None
    if solves > 5e12:
        return {**out, "gains": None, "vmodel": None, "chi2": None, "state": None}
    pi, pj, pt, tp = _pairs(s["sel"])
    V = sums / tp
    g = s["gains"].to(torch.complex128)
    cnt = torch.zeros(s["sel"].n_ubl, dtype=torch.float64, device=DEV).index_add_(0, pt, torch.ones_like(tp))
    V0 = torch.zeros(V.shape[0], s["sel"].n_ubl, dtype=torch.complex128, device=DEV).index_add_(1, pt, V / (g[:, pi] * g[:, pj].conj())) / cnt
    return {**out, **_exact_calibrate(sums, autos, s["sel"], g, V0)}
