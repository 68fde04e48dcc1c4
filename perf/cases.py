"""Measured cases of the coherent-fitness library: what a search program asks of it, through its
public calls, on one GPU.

A case is a dict of plain values: the call, the form (precision), the network and segment, the band
and the batch. `prepare` synthesises what a program has in hand before the call (coloured Gaussian
noise with one injected inspiral per segment, particles, and the context made from them), `run` is
one call, `exact` the same quantities from their definitions in 64-bit torch, `work` the bytes and
operations the call cannot do without.

The FP32 form's Gamma^2 are FP32 numbers that the call widens into a binary64 array: `run` returns
them as FP32, which loses nothing. Gradients and the other forms' results stay binary64.
"""

import math

import numpy as np
import torch

import paper_2002_02150_gb300 as fc

C_LIGHT = 299792458.0
T_SUN = 4.925490947641267e-06          # G Msun / c^3 [s]

# approximate positions and arm bearings of the network (latitude, longitude, x and y arm bearings
# from North; degrees)
SITES = ((46.455147, -119.407656, 324.0, 234.0), (30.562894, -90.774242, 252.2835, 162.2835),
         (43.631414, 10.504497, 19.4326, 289.4326), (36.4119, 137.3056, 60.3964, 150.3964))


def _segment(log_n, n_samples, fs, f_low, f_high, n_det=4):
    return dict(log_n=log_n, n_samples=n_samples, fs=fs, f_low=f_low, f_high=f_high, n_det=n_det)


# 64 s at 1024 Hz (N = 2^16); 60 min at 2048 Hz zero-padded to 2^23, with the band from 30 Hz and
# with the paper's own from 10 Hz; 15 min at 2048 Hz padded to 2^21 with three detectors; a short
# ragged segment padded to 4096
SEG_64S = _segment(16, 65536, 1024.0, 60.0, 500.0)
SEG_60MIN = _segment(23, 7372800, 2048.0, 30.0, 1000.0)
SEG_60MIN_FSTAR10 = _segment(23, 7372800, 2048.0, 10.0, 1000.0)
SEG_15MIN = _segment(21, 1843200, 2048.0, 30.0, 1000.0, n_det=3)
SEG_SHORT = _segment(12, 3000, 512.0, 80.0, 250.0, n_det=3)


def listed():
    return [
        # a host program asks for one point (numpy in, numpy out): launches and latency
        dict(name="one_64s_host", call="fitness", form="fp32", memory="host", particles=1, **SEG_64S),
        # a stream analysis with a fixed memory footprint evaluates a small batch on a short segment
        dict(name="noalloc_short", call="noalloc", form="fp32", particles=24, **SEG_SHORT),
        # one swarm of 40 particles on 64 s, the ordinary step of a program that drives its own search
        dict(name="swarm_64s", call="fitness", form="fp32", particles=40, **SEG_64S),
        # the library's own search, 8 runs of 40 particles (its first iterations: their cost is the same)
        dict(name="search_64s", call="search", form="fp32", runs=8, particles=40, iterations=12, **SEG_64S),
        # background from time-shifted copies of a segment: contexts made, searched together, released
        dict(name="slides_64s", call="slides", form="fp32", slides=4, runs=2, particles=40, iterations=6, **SEG_64S),
        # 15 min, three detectors, an odd batch that spans two of the library's chunks
        dict(name="batch_15min", call="fitness", form="fp32", particles=77, **SEG_15MIN),
        # one point of a 60-min segment in the paper's band (following up a candidate)
        dict(name="one_60min", call="fitness", form="fp32", particles=1, **SEG_60MIN_FSTAR10),
        # 8 runs x 40 particles on 60 min: one iteration of the full search, the largest call
        dict(name="swarms_60min", call="fitness", form="fp32", particles=320, **SEG_60MIN),
        # the binary64 form: checking a swarm in full precision
        dict(name="fp64_64s", call="fitness", form="fp64", particles=40, **SEG_64S),
        # the float-float form: each run's best point of a 60-min search in binary64-class accuracy
        dict(name="ff_60min", call="fitness", form="ff", particles=8, **SEG_60MIN),
        # differentiation through torch: forward and backward of a swarm on 64 s
        dict(name="autograd_64s", call="autograd", form="fp32", particles=40, **SEG_64S),
        # the adjoint at the best points of the 8 runs of a 60-min search
        dict(name="gradient_60min", call="gradient", form="fp32", particles=8, **SEG_60MIN),
    ]


def draw(rng):
    call = rng.choice(["fitness"] * 6 + ["noalloc", "search", "slides", "autograd", "autograd", "gradient", "gradient"])
    form = "fp32" if call in ("search", "slides") else rng.choice(["fp32"] * 4 + ["fp64", "ff"])
    top = {"search": 18, "slides": 18, "noalloc": 20 if form == "fp32" else 19}.get(call, 23)
    log_n = rng.randint(12, top)
    n = 1 << log_n
    fs = rng.choice([512.0, 1024.0, 2048.0])
    # from just over half of the transform length (ragged) to all of it
    n_samples = n if rng.random() < 0.2 else rng.randint(n // 2 + 1, n)
    # the 1.4 + 1.4 Msun signal takes at most 0.4 of the segment
    f_fit = 10.0 * (_chirp_times(1.4, 1.4, 10.0)[0] / (0.4 * n_samples / fs)) ** 0.375
    f_low = round(max(10.0, f_fit) * rng.uniform(1.0, 1.5), 3)
    f_high = round(fs * rng.uniform(0.4, 0.495), 3)
    case = dict(call=call, form=form, log_n=log_n, n_samples=n_samples, fs=fs, f_low=f_low, f_high=f_high,
                # (one detector has no gradient: its projection has rank one)
                n_det=rng.choice([2, 3, 4, 4] if call in ("gradient", "autograd") else [1, 2, 3, 4, 4]))
    if call in ("search", "slides"):
        case.update(runs=rng.randint(1, 4), particles=rng.randint(20, 60), iterations=rng.randint(3, 8))
        if call == "slides":
            case.update(slides=rng.randint(2, 5))
        return case
    # points of transform the call may cover: the largest listed call's (the slower forms less)
    points = {"fp32": 320 << 23, "ff": 32 << 23, "fp64": 6 << 23}[form]
    if call in ("gradient", "autograd"):
        points = min(points, 8 << 23)
    most = max(1, min(640, points >> log_n))
    if call == "gradient":
        case["particles"] = rng.randint(1, min(most, 64))
    else:
        case["particles"] = min(most, int(math.exp(rng.uniform(0.0, math.log(most + 1)))))
    if call == "fitness" and rng.random() < 0.3:
        case["memory"] = "host"
    return case


# ------------------------------------------------------------------------------------------
# synthetic inputs
# ------------------------------------------------------------------------------------------

def _chirp_times(m1, m2, f_star):
    m, eta = (m1 + m2) * T_SUN, m1 * m2 / (m1 + m2) ** 2
    x = math.pi * m * f_star
    return 5.0 / (256.0 * math.pi * f_star * eta) * x ** (-5.0 / 3.0), 1.0 / (8.0 * f_star * eta) * x ** (-2.0 / 3.0)


def _chirp_box(f_star):
    """The rectangle (tau0, tau1.5) of component masses 1..3 Msun."""
    t0lo, t15lo = _chirp_times(3.0, 3.0, f_star)
    t0hi, t15hi = _chirp_times(1.0, 1.0, f_star)
    return t0lo, t0hi, t15lo, t15hi


def _detectors(n_det):
    """(D, 9): position, x arm, y arm (earth-fixed; WGS-84 ellipsoid, horizontal arms)."""
    rows = []
    for lat, lon, bx, by in SITES[:n_det]:
        la, lo = math.radians(lat), math.radians(lon)
        f = 1.0 / 298.257223563
        e2 = f * (2.0 - f)
        r = 6378137.0 / math.sqrt(1.0 - e2 * math.sin(la) ** 2)
        pos = [r * math.cos(la) * math.cos(lo), r * math.cos(la) * math.sin(lo), r * (1.0 - e2) * math.sin(la)]
        east = np.array([-math.sin(lo), math.cos(lo), 0.0])
        north = np.array([-math.sin(la) * math.cos(lo), -math.sin(la) * math.sin(lo), math.cos(la)])
        arms = [math.sin(math.radians(b)) * east + math.cos(math.radians(b)) * north for b in (bx, by)]
        rows.append(np.concatenate([pos] + [a / np.linalg.norm(a) for a in arms]))
    return np.array(rows)


def _psd(f):
    """Analytic fit to the aLIGO design sensitivity (one-sided, 1/Hz)."""
    x = f / 215.0
    return 1e-49 * (x ** -4.14 - 5.0 * x ** -2 + 111.0 * (1.0 - x ** 2 + 0.5 * x ** 4) / (1.0 + 0.5 * x ** 2))


def _band(case):
    """First and last template bin: f_low < k fs / N <= f_high, 0 < k < N/2."""
    n = 1 << case["log_n"]
    k = np.arange(n // 2 + 1)
    inside = (k * case["fs"] > case["f_low"] * n) & (k * case["fs"] <= case["f_high"] * n) & (k > 0) & (k < n // 2)
    return int(np.argmax(inside)), int(n // 2 - np.argmax(inside[::-1]))


def _coefficients(tau0, tau15, f_star):
    """Turns of the 2PN stationary phase in phi^-5/3, phi^-1, phi^-2/3, phi^-1/3, phi = f / f_star."""
    x = 5.0 * tau15 / (32.0 * math.pi * tau0)
    eta = x ** (-2.0 / 3.0) / (8.0 * f_star * tau15)
    tau1 = 5.0 / (192.0 * math.pi * f_star * eta * x) * (743.0 / 336.0 + 11.0 * eta / 4.0)
    tau2 = 5.0 / (128.0 * math.pi * f_star * eta * x ** (1.0 / 3.0)) * (
        3058673.0 / 1016064.0 + 5429.0 * eta / 1008.0 + 617.0 * eta ** 2 / 144.0)
    return 0.6 * f_star * tau0, f_star * tau1, -1.5 * f_star * tau15, 3.0 * f_star * tau2


def _sky(det, alpha, delta):
    """Antenna patterns (D, 2) at psi = 0 and arrival delays (D,) of a direction (torch scalars)."""
    ca, sa, cd, sd = torch.cos(alpha), torch.sin(alpha), torch.cos(delta), torch.sin(delta)
    zero = torch.zeros_like(ca)
    n = torch.stack([cd * ca, cd * sa, sd])
    bx, by = torch.stack([sa, -ca, zero]), torch.stack([-sd * ca, -sd * sa, cd])
    r, xa, ya = det[:, 0:3], det[:, 3:6], det[:, 6:9]
    x_x, x_y, y_x, y_y = xa @ bx, xa @ by, ya @ bx, ya @ by
    return torch.stack([0.5 * (x_x ** 2 - x_y ** 2 - y_x ** 2 + y_y ** 2), x_x * x_y - y_x * y_y], dim=1), -(r @ n) / C_LIGHT


def _phase_turns(coef, phi):
    return coef[0] * phi ** (-5.0 / 3.0) + coef[1] / phi + coef[2] * phi ** (-2.0 / 3.0) + coef[3] * phi ** (-1.0 / 3.0)


def _inputs(case, seed):
    """Everything made from the seed: detector table, PSD, time series, particles, lags."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    h = np.random.Generator(np.random.Philox(key=[int(seed) & 0xFFFFFFFFFFFFFFFF, 7]))
    n, fs, d = 1 << case["log_n"], case["fs"], case["n_det"]
    det = _detectors(d)
    k_lo, k_hi = _band(case)
    f = torch.arange(k_lo, k_hi + 1, device=dev, dtype=torch.float64) * (fs / n)
    s = _psd(f)
    # an inspiral of 1.2..1.6 Msun components, SNR 8..14, coalescing late enough to lie in the segment
    alpha, delta = h.uniform(0.0, 2.0 * math.pi), math.asin(h.uniform(-1.0, 1.0))
    tau0, tau15 = _chirp_times(h.uniform(1.2, 1.6), h.uniform(1.2, 1.6), case["f_low"])
    tc = int(case["n_samples"] * h.uniform(0.7, 0.95))
    u, delay = _sky(torch.tensor(det, device=dev), *(torch.tensor(v, device=dev, dtype=torch.float64) for v in (alpha, delta)))
    cos_i, psi = h.uniform(-1.0, 1.0), h.uniform(0.0, math.pi)
    rot = torch.tensor([[math.cos(2 * psi), -math.sin(2 * psi)], [math.sin(2 * psi), math.cos(2 * psi)]], device=dev, dtype=torch.float64)
    up = u @ rot
    turns = torch.frac(f * (tc / fs)) + _phase_turns(_coefficients(tau0, tau15, case["f_low"]), f / case["f_low"]) + h.uniform()
    spec = torch.zeros((d, n // 2 + 1), device=dev, dtype=torch.complex128)
    resp = [torch.complex(up[i, 0] * (0.5 * (1.0 + cos_i ** 2)), -up[i, 1] * cos_i) for i in range(d)]
    power = sum(float(abs(c) ** 2) for c in resp) * float(4.0 * (fs / n) * torch.sum(f ** (-7.0 / 3.0) / s))
    amp = h.uniform(8.0, 14.0) / math.sqrt(power)
    for i in range(d):
        noise = torch.randn((2, f.numel()), generator=g, device=dev, dtype=torch.float64) * torch.sqrt(s * (n / fs) / 4.0)
        th = -2.0 * math.pi * (turns + f * delay[i])
        spec[i, k_lo:k_hi + 1] = torch.complex(noise[0], noise[1]) + (amp * resp[i]) * f ** (-7.0 / 6.0) * torch.polar(torch.ones_like(th), th)
    data = (torch.fft.irfft(spec, n=n, dim=1) * fs)[:, :case["n_samples"]].contiguous()
    del spec
    grid = torch.arange(n // 2 + 1, device=dev, dtype=torch.float64) * (fs / n)
    psd = _psd(grid)
    psd[0] = psd[1]
    # particles: over the whole sky and chirp-time box, a quarter of them gathered around the signal
    # (gradients: all of them, at the signal's lag give or take a sample)
    p = case["particles"]
    t0lo, t0hi, t15lo, t15hi = _chirp_box(case["f_low"])
    theta = np.stack([h.uniform(0.0, 2.0 * math.pi, p), np.arcsin(h.uniform(-1.0, 1.0, p)), h.uniform(t0lo, t0hi, p),
                      h.uniform(t15lo, t15hi, p)], axis=1)
    near = np.stack([alpha + h.normal(0.0, 0.05, p), delta + h.normal(0.0, 0.05, p), tau0 * (1.0 + h.normal(0.0, 1e-4, p)),
                     tau15 * (1.0 + h.normal(0.0, 1e-3, p))], axis=1)
    gathered = np.ones(p, dtype=bool) if case["call"] == "gradient" else np.arange(p) % 4 == 3
    theta[gathered] = near[gathered]
    lags = np.clip(tc + h.integers(-1, 2, p), 0, case["n_samples"] - 1)
    return dict(det=det, psd=psd.repeat(d, 1), data=data, theta=np.ascontiguousarray(theta), lags=lags.astype(np.int64))


def _box(case):
    return (0.0, 2.0 * math.pi, -0.5 * math.pi, 0.5 * math.pi) + _chirp_box(case["f_low"])


# ------------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------------

def prepare(case, seed):
    s = _inputs(case, seed)
    segment = dict(n_fft=1 << case["log_n"], fs=case["fs"], f_low=case["f_low"], f_high=case["f_high"], precision=case["form"])
    state = dict(case=case, det=s["det"], psd=s["psd"], data=s["data"], segment=segment)
    call = case["call"]
    if call in ("search", "slides"):
        state["cfg"] = fc.pso_config(n_runs=case["runs"], n_particles=case["particles"], n_iter=case["iterations"],
                                     seed=seed, box=_box(case))
    if call == "slides":
        step = int(max(1, min(10 * case["fs"], case["n_samples"] // (4 * case["slides"] + 1))))
        state["shifts"] = np.arange(case["slides"])[:, None] * np.arange(case["n_det"])[None, :] * step
        return state
    state["ctx"] = fc.fcas_create(s["det"], s["psd"], s["data"], **segment)
    del state["psd"], state["data"]       # the context keeps what it needs
    if call == "search":
        return state
    if case.get("memory") == "host":
        state["theta"] = s["theta"]
        return state
    state["theta"] = torch.tensor(s["theta"], device="cuda")
    if call == "gradient":
        state["lags"] = torch.tensor(s["lags"], device="cuda")
    if call == "autograd":
        state["theta"].requires_grad_(True)
    if call == "noalloc":
        state["fitness"] = torch.empty(case["particles"], dtype=torch.float64, device="cuda")
        state["tc"] = torch.empty(case["particles"], dtype=torch.int64, device="cuda")
    return state


def _statistic(case, fitness):
    """Gamma^2 in the form's own type (FP32 numbers in the FP32 form)."""
    if case["form"] != "fp32":
        return fitness
    return fitness.to(torch.float32) if isinstance(fitness, torch.Tensor) else fitness.astype(np.float32)


def _results(case, runs):
    return dict(fitness=_statistic(case, np.array([r["fitness"] for r in runs])), theta=np.array([r["theta"] for r in runs]),
                tc=np.array([r["tc"] for r in runs]), evaluations=np.array([r["evaluations"] for r in runs]))


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "fitness":
        fitness, tc = fc.fcas_fitness(state["ctx"], state["theta"])
        return dict(fitness=_statistic(case, fitness), tc=tc)
    if call == "noalloc":
        fitness, tc = fc.fcas_fitness_noalloc(state["ctx"], state["theta"], state["fitness"], state["tc"])
        return dict(fitness=_statistic(case, fitness), tc=tc)
    if call == "gradient":
        return dict(gradient=fc.fcas_gradient(state["ctx"], state["theta"], state["lags"]))
    if call == "autograd":
        theta = state["theta"]
        theta.grad = None
        fitness, tc = fc.coherent_fitness(state["ctx"], theta)
        fitness.sum().backward()
        return dict(fitness=_statistic(case, fitness.detach()), tc=tc, gradient=theta.grad)
    if call == "search":
        return _results(case, fc.fcas_search(state["ctx"], state["cfg"]))
    best, slides = fc.time_slide_background(state["det"], state["psd"], state["data"], shifts=state["shifts"],
                                            cfg=state["cfg"], **state["segment"])
    return dict(best=_statistic(case, best), **_results(case, [r for s in slides for r in s]))


# ------------------------------------------------------------------------------------------
# the same quantities in 64 bits, and the work
# ------------------------------------------------------------------------------------------

def exact(case, seed):
    """Gamma^2, its argmax and its gradient from their definitions, complex128 torch. None for the
    searches: a swarm's path has no value without the swarm."""
    if case["call"] in ("search", "slides"):
        return None
    s = _inputs(case, seed)
    dev = s["data"].device
    n, fs, f_star = 1 << case["log_n"], case["fs"], case["f_low"]
    df = fs / n
    k_lo, k_hi = _band(case)
    band = slice(k_lo, k_hi + 1)
    k = torch.arange(k_lo, k_hi + 1, device=dev, dtype=torch.int64)
    f = k.to(torch.float64) * df
    det = torch.tensor(s["det"], device=dev)
    psd = s["psd"][:, band]
    y = torch.stack([torch.fft.rfft(x, n=n)[band] for x in s["data"]]) / fs / psd
    y = 4.0 * df * y * f ** (-7.0 / 6.0) * complex(math.sqrt(0.5), -math.sqrt(0.5))
    sigma2 = 4.0 * df * torch.sum(f ** (-7.0 / 3.0) / psd, dim=1)
    s["data"] = s["psd"] = None
    phi = f / f_star

    def network(th):
        """G^-1 and the two antenna-weighted correlation spectra."""
        u, delay = _sky(det, th[0], th[1])
        turns = _phase_turns(_coefficients(th[2], th[3], f_star), phi)
        p = 0.0
        for i in range(case["n_det"]):
            a = 2.0 * math.pi * (turns + f * delay[i])
            q = y[i] * torch.polar(torch.ones_like(a), a)
            p = p + u[i].to(torch.complex128)[:, None] * q[None, :]
        gram = (u * sigma2[:, None]).T @ u
        return gram, p

    def inverse(gram):
        return torch.linalg.pinv(gram, hermitian=True, rtol=2.5e-13)

    theta = torch.tensor(s["theta"], device=dev)
    fitness = torch.empty(case["particles"], dtype=torch.float64, device=dev)
    tc = torch.empty(case["particles"], dtype=torch.int64, device=dev)
    gradient = torch.empty((case["particles"], 4), dtype=torch.float64, device=dev)
    lags = torch.tensor(s["lags"], device=dev)
    for j in range(case["particles"]):
        if case["call"] != "gradient":
            gram, p = network(theta[j])
            root = torch.linalg.cholesky(inverse(gram)) if case["n_det"] > 1 else None
            full = torch.zeros(n, dtype=torch.complex128, device=dev)
            w = []
            for a in range(2):
                full[band] = p[a]
                w.append(torch.fft.ifft(full)[:case["n_samples"]] * n)
            if root is not None:
                total = (root[0, 0] * w[0] + root[1, 0] * w[1]).abs() ** 2 + (root[1, 1] * w[1]).abs() ** 2
            else:
                e = inverse(gram)
                total = (e[0, 0] * w[0].abs() ** 2 + e[1, 1] * w[1].abs() ** 2 + 2.0 * e[0, 1] * (w[0] * w[1].conj()).real)
            tc[j] = torch.argmax(total)
            fitness[j] = total[tc[j]]
            lags[j] = tc[j]
        if case["call"] in ("gradient", "autograd"):
            th = theta[j].clone().requires_grad_(True)
            gram, p = network(th)
            # exact turns of e^{2 pi i k t / N}
            shift = 2.0 * math.pi * ((k * lags[j]) % n).to(torch.float64) / n
            w = (p * torch.polar(torch.ones_like(shift), shift)).sum(dim=1)
            inv = torch.linalg.inv(gram)
            quad = (w.real @ inv @ w.real) + (w.imag @ inv @ w.imag)
            gradient[j] = torch.autograd.grad(quad, th)[0]
    if case["call"] == "gradient":
        return dict(gradient=gradient)
    out = dict(fitness=fitness, tc=tc)
    if case["call"] == "autograd":
        out["gradient"] = gradient
    return out


def work(case):
    n, d = 1 << case["log_n"], case["n_det"]
    k_lo, k_hi = _band(case)
    band = k_hi - k_lo + 1
    p = case["particles"]
    # one evaluation: the network-weighted spectrum (per detector and bin a product with the delay
    # phasor and two weighted sums; the chirp phase and its two products), two transforms, Gamma^2
    one = 10.0 * n * case["log_n"] + (14.0 * d + 20.0) * band + 4.0 * n
    value = 8.0 if case["form"] == "fp32" else 16.0
    spectrum = d * band * value
    # one gradient: per detector and bin the phased value and its six weighted sums
    grad = d * band * 45.0
    call = case["call"]
    if call in ("fitness", "noalloc"):
        return dict(bytes=spectrum + 48.0 * p, flops=p * one)
    if call == "gradient":
        return dict(bytes=spectrum + 72.0 * p, flops=p * grad)
    if call == "autograd":
        return dict(bytes=spectrum + 80.0 * p, flops=p * (one + grad))
    rows = case["runs"] * p * case["iterations"]
    if call == "search":
        return dict(bytes=spectrum, flops=rows * one)
    # per slide: the real transform of each detector's series, whitening, then the search
    made = d * (2.5 * n * case["log_n"] + 12.0 * band)
    return dict(bytes=8.0 * d * (case["n_samples"] + band), flops=case["slides"] * (made + rows * one))
