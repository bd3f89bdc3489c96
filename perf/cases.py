"""Performance cases of the library: the calls its users make, at the sizes they make them.

A case is one call path (`kind`) at one size:

  device   fg21_loglike_batch_device: parameters and logL on the GPU
  host     fg21_loglike_batch: parameters and logL in host arrays, as a CPU sampler holds them
  graph    fg21_graph_launch: the captured evaluation of one or several models (`models` > 1: an
           uneven batch, every model with its own size)
  serve    fg21_serve_submit / fg21_serve_wait: requests of several runs through the serving loop
  noise    fg21_noise_loglike and fg21_noise_q: the accuracy criterion's likelihood distribution
  build    fg21_build_regions and the model's arrays

Sizes are those of the repository's workloads (paper_2603_13196_gb300/inputs.py), benchmark and
tests, and odd ones between them.  `points` says where the parameters lie: "prior" (draws from the
prior, as at the start of a run) or "posterior" (within `spread` of one point that the data were made
from, as a converging run proposes).  The skies have 3072 pixels unless the case says otherwise: the
cost of a likelihood does not depend on the pixels.
"""
import math

import numpy as np
import torch

from paper_2603_13196_gb300 import fg21

T_CMB, NU0, NOISE = 2.725, 230.0, 0.025
TROUGH = (0.155, 85.0, 15.0)
LARGEST = 24 * 301 * 100 * 16384      # multiply-adds of the largest likelihood


def _ll(name, kind, N, F, T, P, precision="fp16x3", points="prior", spread=0.0, Na=0):
    return dict(name=name, kind=kind, N=N, Na=Na, F=F, T=T, P=P, precision=precision, points=points, spread=spread)


def listed():
    return [
        # one step of a small run's chains: launch latency (N = 3, one time bin, 64 points)
        _ll("chains_64", "device", 3, 151, 1, 64),
        # a CPU sampler's batch of replacement points, from and to its own host arrays
        _ll("host_500", "host", 14, 151, 10, 500),
        # a mid-size run: 9 regions, 20 bins over 6 h, 4096 points
        _ll("run_4096", "device", 9, 151, 20, 4096),
        # the benchmark observation: 24 regions, 301 channels, 100 bins, 16384 prior draws, as a graph
        _ll("observation_16384", "graph", 24, 301, 100, 16384),
        # the same observation while the run converges: points close together near the posterior
        _ll("posterior_16384", "device", 24, 301, 100, 16384, points="posterior", spread=1e-5),
        # many regions and bins with nothing a multiple of a tile: more than one t-chunk
        _ll("ragged_3001", "device", 41, 211, 217, 3001),
        # the joint amplitude / spectral-index model: 12 x 2 components with gains
        _ll("amplitude_8192", "device", 12, 301, 50, 8192, Na=2),
        # 32 observations of uneven N, T and P in one launch
        dict(name="uneven_32", kind="graph", models=32, F=151, N_lo=4, N_hi=30, T_lo=1, T_hi=60, P_lo=256, P_hi=8192,
             precision="fp16x3"),
        # the maximum-likelihood search over region counts: the FP32 reference-subtracted form
        _ll("search_fp32_4096", "device", 20, 151, 20, 4096, precision="fp32_delta"),
        # concurrent runs of different N and T sending requests to the serving loop
        dict(name="serve_24", kind="serve", runs=8, requests=24, F=151, P_lo=128, P_hi=4096),
        # the accuracy criterion's noise-only likelihoods at the benchmark observation's cells
        dict(name="noise_65536", kind="noise", n_cells=30100, K=65536, n_bar=16),
        # a new observation: partition and response functions of a 12288-pixel sky
        dict(name="build_12288", kind="build", npix=12288, N=9, F=151, T=20),
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["device", "device", "device", "graph", "graph", "host", "multi", "serve", "noise", "build"])
    F = rng.choice([51, 101, 151, 151, 203, 301])
    if kind == "noise":
        return dict(kind="noise", n_cells=_log(rng, 151, 30100), K=_log(rng, 1000, 65536), n_bar=rng.randint(1, 30))
    if kind == "build":
        return dict(kind="build", npix=_log(rng, 768, 12288), N=rng.randint(1, 30), F=rng.choice([51, 101, 151]),
                    T=_log(rng, 1, 20))
    if kind == "serve":
        return dict(kind="serve", runs=rng.randint(3, 10), requests=rng.randint(8, 32), F=151,
                    P_lo=128, P_hi=_log(rng, 1000, 4096))
    if kind == "multi":
        return dict(kind="graph", models=rng.randint(2, 32), F=rng.choice([51, 101, 151]), N_lo=rng.randint(2, 6),
                    N_hi=rng.randint(8, 40), T_lo=1, T_hi=rng.randint(8, 72), P_lo=rng.randint(32, 256),
                    P_hi=_log(rng, 512, 8192), precision="fp16x3")
    precision = rng.choice(["fp16x3"] * 8 + ["bf16x3", "fp32_delta", "fp32_delta"])
    N = rng.randint(2, 45) if rng.random() < 0.9 else rng.randint(46, 62)
    T = _log(rng, 1, 220)
    Na = 0
    if precision == "fp16x3" and rng.random() < 0.2:
        Na, N = rng.randint(1, 4), rng.randint(2, 12)
    comps = N * max(Na, 1)
    top = min(16384, max(64, LARGEST // (3 * comps * F * T)))
    P = _log(rng, 32, top)
    points = rng.choice(["prior", "posterior"])
    return dict(kind=kind, N=N, Na=Na, F=F, T=T, P=P, precision=precision, points=points,
                spread=10.0 ** rng.randint(-6, -2) if points == "posterior" else 0.0)


# ------------------------------------------------------------------ inputs
class _Record:
    def __init__(self, **kw):
        self.__dict__.update(kw)


def _rng(seed, stream):
    return np.random.default_rng([int(seed), stream])


def _sky(npix, seed):
    """Near-equal-area pixels, a bright band with scatter, spectral indices around 2.55."""
    k = np.arange(npix) + 0.5
    z = 1.0 - 2.0 * k / npix
    phi = math.pi * (1.0 + math.sqrt(5.0)) * k
    s = np.sqrt(np.maximum(0.0, 1.0 - z * z))
    dirs = np.stack([s * np.cos(phi), s * np.sin(phi), z], axis=1)
    r = _rng(seed, 1)
    t230 = (150.0 + 3000.0 * np.exp(-np.abs(np.arcsin(z)) / math.radians(8.0))) * np.exp(0.3 * r.standard_normal(npix))
    beta = 2.55 + 0.1 * np.sin(np.arctan2(dirs[:, 1], dirs[:, 0])) + 0.02 * r.standard_normal(npix)
    return _Record(dirs=dirs, t230=t230, beta=beta)


def _obs(F, T, seed):
    """F channels of 50-200 MHz, T bins of up to 12 h from a random hour, a beam cos^p with p(nu) oscillating."""
    nu = np.linspace(50.0, 200.0, F)
    r = _rng(seed, 2)
    start, window = r.uniform(0.0, 24.0), 0.0 if T == 1 else r.choice([6.0, 12.0])
    ang = (start + (np.arange(T) + 0.5) * window / T) * (2.0 * math.pi / 24.0)
    lat = math.radians(-30.7)
    zen = np.stack([math.cos(lat) * np.cos(ang), math.cos(lat) * np.sin(ang), np.full(T, math.sin(lat))], axis=1)
    tilt = math.radians(62.9)          # the celestial pole's distance from the band's pole
    rot = np.array([[1, 0, 0], [0, math.cos(tilt), -math.sin(tilt)], [0, math.sin(tilt), math.cos(tilt)]])
    zen = zen @ rot.T
    zen /= np.linalg.norm(zen, axis=1, keepdims=True)
    return _Record(nu=nu, zenith=zen, beam_p=1.5 + 0.3 * np.sin(2.0 * math.pi * nu / 40.0), nu0=NU0, t_cmb=T_CMB)


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _beams(sky, obs):
    """Per channel, the beam towards every pixel in every bin: [T, npix] FP64."""
    c = (_dev(obs.zenith)[:, :, None] * _dev(sky.dirs).T[None]).sum(1)
    up = c > 0
    lc = torch.where(up, c, torch.ones_like(c)).log()
    for p in obs.beam_p.tolist():
        yield torch.where(up, 2.0 * (p + 1.0) * torch.exp(p * lc), torch.zeros_like(lc))


def _trough(nu, a, c, s):
    return a * torch.exp(-((nu - c) ** 2) / (2.0 * s * s))


def _observed(sky, obs, seed):
    """The data: the sky pixel by pixel, a trough and 25 mK of noise, [F, T]."""
    t, b = _dev(sky.t230), _dev(sky.beta)
    rows = []
    for d, nu in zip(_beams(sky, obs), obs.nu.tolist()):
        rows.append((d * ((t - T_CMB) * torch.exp(-b * math.log(nu / NU0)) + T_CMB)).mean(1))
    T21 = _trough(_dev(obs.nu), *TROUGH)[:, None]
    return torch.stack(rows) + T21 + NOISE * _dev(_rng(seed, 3).standard_normal((len(obs.nu), len(obs.zenith))))


def _weights(sky, obs):
    """Each pixel's importance: its share of the beam-weighted sky, averaged over channels and bins."""
    t, b = _dev(sky.t230), _dev(sky.beta)
    w = torch.zeros_like(t)
    for d, nu in zip(_beams(sky, obs), obs.nu.tolist()):
        x = d * ((t - T_CMB) * torch.exp(-b * math.log(nu / NU0)) + T_CMB)
        w += (x / x.sum(1, keepdim=True)).sum(0)
    return (w / (len(obs.nu) * len(obs.zenith))).cpu().numpy()


def _recursive(field, w, N):
    """(labels, edges): the interval of largest mass halved until there are N, the lowest of equals first."""
    def mass(a, b, closed):
        m = ((field >= a) if closed else (field > a)) & (field <= b)
        return math.fsum(w[m])

    lo, hi = float(field.min()), float(field.max())
    regions = [[lo, hi, True, mass(lo, hi, True)]]
    while len(regions) < N:
        r = max(regions, key=lambda x: (x[3], -x[0]))
        mid = 0.5 * (r[0] + r[1])
        up = [mid, r[1], False, mass(mid, r[1], False)]
        r[1], r[3] = mid, mass(r[0], mid, r[2])
        regions.append(up)
    edges = np.array([lo] + sorted(r[1] for r in regions))
    return np.searchsorted(edges[1:N], field, side="left").astype(np.int32), edges


def _responses(sky, obs, comp, n):
    """A [n, F, T] and B [F, T] of the components `comp` (one per pixel)."""
    one = torch.zeros((sky.t230.shape[0], n), dtype=torch.float64, device="cuda")
    one[torch.arange(len(comp)), torch.as_tensor(comp, dtype=torch.long)] = 1.0
    one = one * (_dev(sky.t230) - T_CMB)[:, None] / len(comp)
    A, B = [], []
    for d in _beams(sky, obs):
        A.append((d @ one).T)
        B.append(d.mean(1))
    return torch.stack(A, 1), torch.stack(B)


def _parts(c, seed):
    """The sky, the observation and, in FP64 by torch, the labels, edges, A and B of a likelihood or build case."""
    sky, obs = _sky(c.get("npix", 3072), seed), _obs(c["F"], c["T"], seed)
    w = _weights(sky, obs)
    lab, edges = _recursive(sky.beta, w, c["N"])
    comp, n = lab, c["N"]
    if c.get("Na"):
        lab_a, _ = _recursive(np.log(sky.t230), w, c["Na"])
        comp, n = lab_a * c["N"] + lab, c["N"] * c["Na"]
    A, B = _responses(sky, obs, comp, n)
    return sky, obs, lab, edges, A, B


def _powers(c, obs, th):
    """The weight of every component for every point, channel by channel: [P, components]."""
    N, Na = c["N"], c["Na"]
    for nu in obs.nu.tolist():
        w = torch.exp(-th[:, :N] * math.log(nu / NU0))
        yield (th[:, N:N + Na, None] * w[:, None, :]).reshape(len(th), -1) if Na else w


def _params(c, seed, stream=4):
    """Parameter rows [P, N + Na + 4] of a case, and the truth they lie around (posterior points)."""
    r, N, Na, P = _rng(seed, stream), c["N"], c.get("Na", 0), c["P"]
    if c.get("points") == "posterior":
        truth = np.concatenate([r.uniform(2.5, 2.7, N), r.uniform(0.95, 1.05, Na), TROUGH, [NOISE]])
        th = np.repeat(truth[None], P, 0)
        th[:, :N] += r.uniform(-c["spread"], c["spread"], (P, N))
        if Na:
            th[:, N:N + Na] *= 1.0 + r.uniform(-c["spread"], c["spread"], (P, Na))
        return th, truth
    cols = [r.uniform(2.45, 3.15, (P, N)), r.uniform(0.9, 1.1, (P, Na)), r.uniform(0.0, 0.25, (P, 1)),
            r.uniform(50.0, 200.0, (P, 1)), r.uniform(5.0, 40.0, (P, 1)), np.exp(r.uniform(math.log(1e-3), math.log(0.1), (P, 1)))]
    return np.concatenate(cols, axis=1), None


def _data(c, seed, sky, obs, A, B, truth):
    if truth is None:
        return _observed(sky, obs, seed)
    th = _dev(truth)[None]
    rows = [w @ A[:, f] for f, w in enumerate(_powers(c, obs, th))]
    noise = _dev(_rng(seed, 3).standard_normal(tuple(B.shape)))
    return torch.cat(rows) + T_CMB * B + _trough(_dev(obs.nu), *TROUGH)[:, None] + NOISE * noise


def _inputs(c, seed):
    """What a likelihood case is made of: sky, observation, data [F, T] and parameter rows."""
    th, truth = _params(c, seed)
    if truth is None:
        sky, obs, A, B = _sky(3072, seed), _obs(c["F"], c["T"], seed), None, None
    else:
        sky, obs, _, _, A, B = _parts(c, seed)
    return sky, obs, _data(c, seed, sky, obs, A, B, truth), th


def _sizes(c, seed):
    """The members of an uneven batch or of a serving mix, as likelihood cases of their own.  Their sizes come
    from the case alone, so that every seed asks for the same work."""
    r = np.random.default_rng([c.get("models", 0), c.get("runs", 0), c["P_hi"], 7])
    if c["kind"] == "graph":
        return [dict(N=int(r.integers(c["N_lo"], c["N_hi"] + 1)), Na=0, F=c["F"], T=int(r.integers(c["T_lo"], c["T_hi"] + 1)),
                     P=int(r.integers(c["P_lo"], c["P_hi"] + 1)), seed=seed * 1000 + k) for k in range(c["models"])]
    runs = [dict(N=(5, 9, 14, 20, 30)[k % 5], Na=0, F=c["F"], T=(1, 10, 50)[k % 3], P=1, seed=seed * 1000 + k)
            for k in range(c["runs"])]
    reqs = [(int(r.integers(0, c["runs"])), int(r.integers(c["P_lo"], c["P_hi"] + 1))) for _ in range(c["requests"])]
    return runs, reqs


def _model(c, sky, obs, data):
    if c.get("Na"):
        m = fg21.fg21_build_regions_ab(sky, obs, c["N"], "recursive", "beam", c["Na"], np.log(sky.t230), "recursive")
    else:
        m = fg21.fg21_build_regions(sky, obs, c["N"], "recursive", "beam")
    fg21.fg21_model_set_data(m, data.cpu().numpy())
    return m


class _State(dict):
    """A case's state; the library's handles are closed in order when it goes."""

    def __del__(self):
        for k in ("server", "graph"):
            if self.get(k) is not None:
                self[k].close()


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "noise":
        mean = -0.5 * c["n_cells"] * (math.log(2.0 * math.pi * NOISE * NOISE) + 1.0)
        bars = mean + math.sqrt(0.5 * c["n_cells"]) * _rng(seed, 5).standard_normal(c["n_bar"])
        return _State(c=c, seed=seed, out=torch.empty(c["K"], dtype=torch.float64, device="cuda"), bars=bars)
    if c["kind"] == "build":
        return _State(c=c, sky=_sky(c["npix"], seed), obs=_obs(c["F"], c["T"], seed))
    if c["kind"] == "serve":
        runs, reqs = _sizes(c, seed)
        models = []
        for r in runs:
            sky, obs, data, _ = _inputs(r, r["seed"])
            models.append(_model(r, sky, obs, data))
        server = fg21.Server(mem_budget_bytes=60 << 30, max_batch_points=65536, max_wait_us=200, max_inflight=2)
        ids = [fg21.fg21_serve_register_run(server, m)[0] for m in models]
        ths = [_params(dict(runs[k], P=P), seed * 1000 + j, 6)[0] for j, (k, P) in enumerate(reqs)]
        return _State(c=c, server=server, models=models, reqs=[(ids[k], th) for (k, _), th in zip(reqs, ths)])
    members = _sizes(c, seed) if c.get("models") else [dict(c, seed=seed)]
    models, ths = [], []
    for k in members:
        sky, obs, data, th = _inputs(k, k["seed"])
        models.append(_model(k, sky, obs, data))
        ths.append(th)
    if c["kind"] == "host":
        return _State(c=c, model=models[0], th=ths[0])
    d_th = [_dev(th) for th in ths]
    outs = [torch.empty(len(th), dtype=torch.float64, device="cuda") for th in ths]
    s = _State(c=c, models=models, th=d_th, out=outs)
    if c["kind"] == "graph":
        torch.cuda.synchronize()
        s["graph"] = fg21.fg21_graph_create_multi(models, [t.data_ptr() for t in d_th], [len(t) for t in d_th],
                                                  [o.data_ptr() for o in outs], c["precision"])
    return s


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "host":
        return fg21.fg21_loglike_batch(state["model"], state["th"], c["precision"])
    if kind == "build":
        m = fg21.fg21_build_regions(state["sky"], state["obs"], c["N"], "recursive", "beam")
        A, B = fg21.fg21_model_get_arrays(m)
        m.close()
        return m.labels, m.edges, A, B
    if kind == "serve":
        s = state["server"]
        sent = [fg21.fg21_serve_submit(s, rid, th) for rid, th in state["reqs"]]
        for ticket, _ in sent:
            if fg21.fg21_serve_wait(s, ticket) != fg21.FG21_OK:
                raise RuntimeError("a request failed")
        return [out for _, out in sent]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "noise":
        fg21.fg21_noise_loglike(c["n_cells"], NOISE, NOISE, c["K"], state["seed"], state["out"].data_ptr(), stream)
        return state["out"], fg21.fg21_noise_q(state["out"].data_ptr(), c["K"], state["bars"], stream)
    if kind == "graph":
        state["graph"].launch(stream)
        return state["out"]
    th, out = state["th"][0], state["out"][0]
    fg21.fg21_loglike_batch_device(state["models"][0], th.data_ptr(), len(th), out.data_ptr(), c["precision"], stream)
    return out


# ------------------------------------------------------------------- work
def _ll_work(N, Na, F, T, P):
    n = N * max(Na, 1)
    return 8.0 * (P * (N + Na + 5) + n * F * T + 2 * F * T), (2.0 * n + 3.0) * F * T * P


def work(case):
    """Bytes: parameters, A, B and data in FP64 read once, logL written once.  Flops: the contraction over the
    components, and the residual and its square, of every point, channel and bin."""
    c = case
    if c["kind"] == "noise":
        # per pair of draws: ten rounds of two 32 x 32 products and a logarithm (about 60 operations)
        return {"bytes": 8.0 * c["K"], "flops": 60.0 * c["K"] * (c["n_cells"] / 2)}
    if c["kind"] == "build":
        # the beam and the two sums it enters, once per pixel, channel and bin (the exponential as 20 operations)
        cells = c["npix"] * c["F"] * c["T"]
        return {"bytes": 8.0 * (5 * c["npix"] + (c["N"] + 1) * c["F"] * c["T"]), "flops": 25.0 * cells}
    if c["kind"] == "serve":
        runs, reqs = _sizes(c, 0)
        parts = [_ll_work(runs[k]["N"], 0, c["F"], runs[k]["T"], P) for k, P in reqs]
    elif c.get("models"):
        parts = [_ll_work(k["N"], 0, k["F"], k["T"], k["P"]) for k in _sizes(c, 0)]
    else:
        parts = [_ll_work(c["N"], c["Na"], c["F"], c["T"], c["P"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------ 64 bits
def _logl(c, obs, data, A, B, th):
    th = _dev(th)
    nf = th.shape[1] - 4
    sig2 = th[:, nf + 3] ** 2
    chi2 = torch.zeros(len(th), dtype=torch.float64, device="cuda")
    for f, w in enumerate(_powers(c, obs, th)):
        t21 = _trough(float(obs.nu[f]), th[:, nf], th[:, nf + 1], th[:, nf + 2])
        chi2 += ((data[f] - T_CMB * B[f])[None] - w @ A[:, f] - t21[:, None]).square().sum(1)
    return -0.5 * (data.numel() * torch.log(2.0 * math.pi * sig2) + chi2 / sig2)


def _member_logl(k, ths):
    """logL in 64 bits of one likelihood case's observation for each set of rows."""
    sky, obs, _, _, A, B = _parts(k, k["seed"])
    _, truth = _params(k, k["seed"])
    data = _data(k, k["seed"], sky, obs, A, B, truth)
    return [_logl(k, obs, data, A, B, th) for th in ths]


def _mulhilo(a, m):
    """High and low 32 bits of a * m for 32-bit values in int64 tensors."""
    lo, hi = a * (m & 0xFFFF), a * (m >> 16)
    s = lo + ((hi & 0xFFFF) << 16)
    return (hi >> 16) + (s >> 32), s & 0xFFFFFFFF


def _philox(j, k, seed):
    """The first two output words of Philox4x32-10 (Salmon et al. 2011), counter (j, k, 0, 0), key `seed`."""
    c0, c1, c2, c3 = j, k, torch.zeros_like(j), torch.zeros_like(j)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mulhilo(c0, 0xD2511F53)
        h1, l1 = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1


def _noise(c, seed):
    n, K = c["n_cells"], c["K"]
    j = torch.arange(n // 2, device="cuda", dtype=torch.int64)[None]
    out = []
    step = max(1, (1 << 26) // max(1, n // 2))
    for k0 in range(0, K, step):
        k = torch.arange(k0, min(K, k0 + step), device="cuda", dtype=torch.int64)[:, None]
        x, _ = _philox(j.expand(len(k), -1), k.expand(-1, n // 2), seed)
        s = (-2.0 * torch.log((x + 1).double() / 4294967296.0)).sum(1)
        if n & 1:
            x, y = _philox(torch.full_like(k[:, 0], n // 2), k[:, 0], seed)
            r2 = -2.0 * torch.log((x + 1).double() / 4294967296.0)
            s += r2 * torch.cos(2.0 * math.pi * (y + 1).double() / 4294967296.0).square()
        out.append(s)
    return -0.5 * (n * math.log(2.0 * math.pi * NOISE * NOISE) + torch.cat(out))


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "noise":
        return _noise(c, seed), None
    if c["kind"] == "build":
        _, _, lab, edges, A, B = _parts(c, seed)
        return lab, edges, A.cpu().numpy(), B.cpu().numpy()
    if c["kind"] == "serve":
        runs, reqs = _sizes(c, seed)
        ths = [_params(dict(runs[k], P=P), seed * 1000 + j, 6)[0] for j, (k, P) in enumerate(reqs)]
        got = [None] * len(reqs)
        for r, member in enumerate(runs):
            mine = [j for j, (k, _) in enumerate(reqs) if k == r]
            for j, v in zip(mine, _member_logl(member, [ths[j] for j in mine])):
                got[j] = v.cpu().numpy()
        return got
    members = _sizes(c, seed) if c.get("models") else [dict(c, seed=seed)]
    got = [_member_logl(k, [_params(k, k["seed"])[0]])[0] for k in members]
    if c["kind"] == "graph":
        return got
    return got[0].cpu().numpy() if c["kind"] == "host" else got[0]
