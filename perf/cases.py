"""The work a user of this package has it do, as cases that can be timed and compared.

A case names an operation and its sizes; prepare() makes what a user's program
holds before the call (cubes, handles, source lists), run() is one pass through
the public entry points, exact() the same outputs in 64 bits by plain torch.
Sizes are those of the repository's own configurations (synth.CONFIGS: 32, 128
and 512 antennas; 16, 128, 256 and 768 channels; 5, 50, 100, 300 and 1000
sources), of its tests (ragged antenna and channel counts) and of bench.py's
gridder and integrator legs; draw() spreads more over the same ranges.

Skies are drawn as the synthetic cadences of the repository are: antennas in a
disc of 750 m, |l|, |m| < 0.3, S^-1.6 fluxes in 1..20 Jy sorted brightest
first, gains I + CN(0, 0.1^2).  The noise is a radio array's: its mean over a
cadence is NOISE_JY on every baseline (an MWA tile pair over 31 MHz and 8 s),
so a single sample carries NOISE_JY sqrt(samples).
"""
import math

import numpy as np
import torch

from paper_1003_5575_gb300 import Gridder, Integrator, Peeler, PeelLoss, integration_lengths

C_LIGHT = 299792458.0
OMEGA_EARTH = 7.2921159e-5      # rad / s
LATITUDE = math.radians(-26.703)
ARCMIN = math.pi / 180.0 / 60.0
NOISE_JY = 0.5
TAU = 2.0 * math.pi


def listed():
    return [
        # One calibrator's gains from averages in hand: the step an interactive user or a
        # pipeline with its own averaging calls, one launch chain, latency only.
        {"name": "solve-128", "op": "solve", "ant": 128, "chan": 128, "time": 8, "src": 1},
        # A test array's cadence (configuration 1): launches and latency.
        {"name": "cadence-32x16", "op": "cadence", "ant": 32, "chan": 16, "time": 8, "src": 5},
        # An odd array with a cut band and few samples: ragged tiles everywhere.
        {"name": "cadence-65x203", "op": "cadence", "ant": 65, "chan": 203, "time": 3, "src": 61},
        # The 128-tile array (configuration 2).
        {"name": "cadence-128x128", "op": "cadence", "ant": 128, "chan": 128, "time": 8, "src": 50},
        # The full array, one 8 s cadence, 1000 sources (configuration 3).
        {"name": "cadence-512x768", "op": "cadence", "ant": 512, "chan": 768, "time": 8, "src": 1000},
        # The same 128-tile cadence in double precision: the comparator a user checks against.
        {"name": "fp64-128x128", "op": "fp64", "ant": 128, "chan": 128, "time": 8, "src": 50},
        # Gains linear in frequency on the 128-tile array.
        {"name": "taylor-128x128", "op": "taylor", "ant": 128, "chan": 128, "time": 8, "src": 50},
        # A gradient step of gains, positions and fluxes (configuration 4).
        {"name": "grad-128x256", "op": "grad", "ant": 128, "chan": 256, "time": 8, "src": 100},
        # The gradient step of the full array (configuration 5).
        {"name": "grad-512x768", "op": "grad", "ant": 512, "chan": 768, "time": 8, "src": 300},
        # Model visibilities of a solved sky (configuration 4's shape).
        {"name": "predict-128x256", "op": "predict", "ant": 128, "chan": 256, "time": 8, "src": 100},
        # The gridder at the paper's shape: one channel of the full array.
        {"name": "grid-1125", "op": "grid", "ant": 512, "chan": 1, "pix": 1125, "rmax": 12.0, "bin": 24, "pol": 4},
        # Half-second samples of the 128-tile array into 8, 4 and 2 s groups.
        {"name": "integrate-128x768", "op": "integrate", "ant": 128, "chan": 768, "time": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _peelable(ant, chan, src, per):
    """A source count that `ant` antennas and `chan` channels can tell apart."""
    return max(1, min(src, ant * chan // per))


def draw(rng):
    op = rng.choice(["cadence"] * 4 + ["taylor", "grad", "grad", "predict", "fp64", "solve", "grid", "integrate"])
    if op == "grid":
        rmax = rng.choice([4.0, 6.0, 7.5, 12.0])
        return {"op": op, "ant": _log(rng, 64, 512), "chan": rng.randint(1, 4), "pix": _log(rng, 300, 1125),
                "rmax": rmax, "bin": max(13, int(math.ceil(rmax)) + rng.randint(0, 12)), "pol": rng.randint(1, 4)}
    if op == "integrate":
        return {"op": op, "ant": _log(rng, 16, 128), "chan": _log(rng, 16, 768), "time": 16}
    if op == "solve":
        return {"op": op, "ant": _log(rng, 16, 512), "chan": rng.randint(64, 128), "time": 4, "src": 1}
    if op in ("fp64", "taylor"):
        ant, chan = _log(rng, 16, 128), _log(rng, 32, 128)
        return {"op": op, "ant": ant, "chan": chan, "time": rng.randint(2, 8),
                "src": _peelable(ant, chan, _log(rng, 1, 50), 400)}
    if op in ("grad", "predict"):
        return {"op": op, "ant": _log(rng, 16, 256), "chan": _log(rng, 16, 768), "time": rng.randint(1, 8),
                "src": _log(rng, 2, 300 if op == "grad" else 100)}
    ant, chan = _log(rng, 16, 512), _log(rng, 16, 768)
    return {"op": op, "ant": ant, "chan": chan, "time": rng.randint(1, 8),
            "src": _peelable(ant, chan, _log(rng, 2, 1000), 200)}


def work(case):
    n_bl = case["ant"] * (case["ant"] - 1) // 2
    op = case["op"]
    if op == "grid":
        n = n_bl * case["chan"]
        return {"bytes": n * (8 + 8 * case["pol"]) + 8 * case["pol"] * case["pix"] ** 2,
                "flops": n * math.pi * case["rmax"] ** 2 * 4 * case["pol"]}
    if op == "integrate":
        return {"bytes": (16 + 4) * n_bl * case["chan"] * 32, "flops": 16 * n_bl * case["chan"] * 8}
    if op == "solve":      # 20 sweeps of two 2x2 complex products a pair, either way round
        return {"bytes": 32 * n_bl + 32 * case["ant"], "flops": 20 * 2 * n_bl * 128}
    n_vis, k = n_bl * case["chan"] * case["time"], case["src"]
    jones = 32 * k * case["ant"]
    if op == "grad":       # model, rotated residual and its frequency-weighted sum
        return {"bytes": 32 * n_vis + 2 * jones, "flops": 80 * n_vis * k}
    if op == "predict":
        return {"bytes": 32 * n_vis + jones, "flops": 32 * n_vis * k}
    if op == "taylor":     # three moments and a model of three terms
        return {"bytes": 64 * n_vis + 2 * jones, "flops": 100 * n_vis * k}
    wide = 2 if op == "fp64" else 1
    return {"bytes": wide * (64 * n_vis + jones), "flops": 64 * n_vis * k}


# -- geometry and sky ---------------------------------------------------------

def _array(case, seed):
    """Antenna uvw [time][ant][3] of a flat disc tracked through 1 s samples, channel
    centres, and the antenna pairs of the baselines in their order."""
    r = np.random.RandomState(seed % (1 << 31))
    rad, ang = 750.0 * np.sqrt(r.random_sample(case["ant"])), TAU * r.random_sample(case["ant"])
    e, n = rad * np.cos(ang), rad * np.sin(ang)
    x, y, z = -math.sin(LATITUDE) * n, e, math.cos(LATITUDE) * n
    sd, cd = math.sin(LATITUDE), math.cos(LATITUDE)
    uvw = np.empty((case.get("time", 1), case["ant"], 3))
    for t in range(uvw.shape[0]):
        sh, ch = math.sin(OMEGA_EARTH * t), math.cos(OMEGA_EARTH * t)
        uvw[t, :, 0] = sh * x + ch * y
        uvw[t, :, 1] = -sd * ch * x + sd * sh * y + cd * z
        uvw[t, :, 2] = cd * ch * x - cd * sh * y + sd * z
    freq = 167e6 + 40e3 * np.arange(case["chan"])
    i, j = np.triu_indices(case["ant"], k=1)
    return uvw, freq, torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda()


def _sources(case, seed):
    r = np.random.RandomState((seed + 1000003) % (1 << 31))
    k = case["src"]
    lm = 0.6 * r.random_sample((k, 2)) - 0.3
    s = (1.0 + r.random_sample(k) * (20.0 ** -0.6 - 1.0)) ** (-1.0 / 0.6)
    return np.concatenate([lm, -np.sort(-s)[:, None]], axis=1)


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000 * int(seed) + stream)
    return g


def _gains(case, gen, slope=False):
    """[src][ant][2][2] gains I + CN(0, 0.1^2), or slopes CN(0, 0.2^2) over the band."""
    j = torch.randn((case["src"], case["ant"], 2, 2), dtype=torch.complex128, device="cuda", generator=gen)
    return 0.2 * j if slope else 0.1 * j + torch.eye(2, device="cuda", dtype=torch.complex128)


def _lmn(src):
    src = torch.as_tensor(src, dtype=torch.float64, device="cuda")
    l, m = src[:, 0], src[:, 1]
    return torch.stack([l, m, torch.sqrt(1.0 - l * l - m * m) - 1.0])


def _herm(a):
    return a.conj().transpose(-1, -2)


def _cis(turns):
    a = (TAU * (turns - torch.round(turns))).to(torch.float32)
    return torch.complex(torch.cos(a), -torch.sin(a))


def _cube(case, arr, src, gain, slope, gen):
    """The sky's visibilities plus noise, complex64 [time][bl][chan][4].  Each baseline's
    channels are 16 q + r, so exp(-2 pi i phase) is a product of a q and an r table and a
    baseline is one small complex matrix product over the sources."""
    uvw, freq, ai, aj = arr
    n_t, n_bl, n_c = uvw.shape[0], ai.shape[0], len(freq)
    n_q = -(-n_c // 16)
    lmn = _lmn(src)
    s = torch.as_tensor(src[:, 2], device="cuda").to(torch.complex64)
    gain = gain.to(torch.complex64)
    terms = [(gain, gain)]
    if slope is not None:
        slope = slope.to(torch.complex64)
        terms += [(gain, slope), (slope, gain), (slope, slope)]
    x = (torch.arange(n_c, device="cuda", dtype=torch.float32) - (n_c - 1) / 2) / n_c
    weight = [None, x, x, x * x]
    dnu = 40e3
    sigma = NOISE_JY * math.sqrt(n_t * n_c)
    vis = torch.empty((n_t, n_bl, n_c, 4), dtype=torch.complex64, device="cuda")
    step = max(1, int(2.5e8 / (len(src) * (64 + n_q) + 80 * n_c)))
    q = 16.0 * torch.arange(n_q, device="cuda", dtype=torch.float64)
    r = torch.arange(16, device="cuda", dtype=torch.float64)
    for b in range(0, n_bl, step):
        i, j = ai[b:b + step], aj[b:b + step]
        m = [torch.einsum("knab,kncb->nkac", p[:, i], o[:, j].conj()).reshape(len(i), len(src), 4) * s[None, :, None]
             for p, o in terms]
        for t in range(n_t):
            ut = torch.as_tensor(uvw[t], device="cuda")
            tau = (ut[i] - ut[j]) @ lmn / C_LIGHT                          # [n][k]
            t1 = _cis((tau * freq[0])[..., None] + (tau * dnu)[..., None] * q)   # [n][k][q]
            t2 = _cis((tau * dnu)[..., None] * r)                          # [n][k][r]
            out = vis[t, b:b + step]
            out.normal_(generator=gen)         # Re and Im each of variance 1/2
            out *= sigma * math.sqrt(2.0)
            for mm, w in zip(m, weight):
                a = (mm[:, :, None, :] * t2[..., None]).reshape(len(i), len(src), 64)
                v = torch.bmm(t1.transpose(1, 2), a).reshape(len(i), 16 * n_q, 4)[:, :n_c]
                out += v if w is None else v * w[None, :, None]
    return vis


def _sky(case, seed):
    arr = _array(case, seed)
    src = _sources(case, seed)
    gen = _generator(seed, 1)
    gain = _gains(case, gen)
    slope = _gains(case, gen, slope=True) if case["op"] == "taylor" else None
    return arr, src, gain, slope, gen


def _averages(case, seed):
    """One source's averages S J_i J_j^H + noise, complex64 [bl][4]."""
    arr, src, gain, _, gen = _sky(case, seed)
    v = src[0, 2] * gain[0][arr[2]] @ _herm(gain[0][arr[3]])
    v = v + NOISE_JY * math.sqrt(2.0) * torch.randn(v.shape, dtype=v.dtype, device="cuda", generator=gen)
    return arr, src, v.reshape(-1, 4).to(torch.complex64)


def _taper(n_tab=1025):
    r = np.linspace(0.0, 1.0, n_tab)
    k = np.i0(8.0 * np.sqrt(np.clip(1.0 - r * r, 0.0, None)))
    return (k - k[-1]) / (k[0] - k[-1])


def _uv_points(case, seed):
    """Pixel coordinates of every baseline at every channel, 21.4 degree field, and values."""
    uvw, freq, ai, aj = _array(case, seed)
    u = torch.as_tensor(uvw[0, :, :2], device="cuda")
    d = u[ai] - u[aj]
    cell = math.radians(21.4)
    xy = torch.cat([d * (f / C_LIGHT * cell) + case["pix"] / 2.0 for f in freq]).to(torch.float32).contiguous()
    vis = torch.randn((xy.shape[0], case["pol"]), dtype=torch.complex64, device="cuda",
                      generator=_generator(seed, 2))
    return xy, vis


def _samples(case, seed):
    uvw, _, ai, _ = _array(case, seed)
    lengths = integration_lengths(uvw[uvw.shape[0] // 2], [699.0, 1398.0], [16, 8, 4])
    fine = torch.randn((16, ai.shape[0], case["chan"], 4), dtype=torch.complex64, device="cuda",
                       generator=_generator(seed, 3))
    return lengths, fine


def _perturbed(case, seed, src):
    """Catalogue positions off by 1 arcmin (Gaussian) in l and in m."""
    r = np.random.RandomState((seed + 2000003) % (1 << 31))
    out = src.copy()
    out[:, :2] += ARCMIN * r.standard_normal((len(src), 2))
    return out


# -- what a user holds, and one pass --------------------------------------------

def prepare(case, seed):
    op = case["op"]
    if op == "grid":
        xy, vis = _uv_points(case, seed)
        g = Gridder(case["pix"], case["rmax"], _taper(), bin=case["bin"], n_pol=case["pol"], max_vis=xy.shape[0])
        grid = torch.empty((case["pol"], case["pix"], case["pix"]), dtype=torch.complex64, device="cuda")
        return {"op": op, "g": g, "xy": xy, "vis": vis, "grid": grid}
    if op == "integrate":
        lengths, fine = _samples(case, seed)
        g = Integrator(16, case["chan"], lengths, n_slot=4)
        out = torch.empty((4,) + tuple(fine.shape[1:]), dtype=torch.complex64, device="cuda")
        return {"op": op, "g": g, "fine": fine, "out": out}
    if op == "solve":
        arr, src, avg = _averages(case, seed)
        return {"op": op, "p": Peeler(arr[0], arr[1], max_sources=1), "avg": avg, "S": float(src[0, 2])}
    arr, src, gain, slope, gen = _sky(case, seed)
    gain64 = gain.reshape(case["src"], case["ant"], 4).to(torch.complex64).contiguous()
    vis = None if op == "predict" else _cube(case, arr, src, gain, slope, gen)
    torch.cuda.empty_cache()            # the library's handle allocates its own memory
    p = Peeler(arr[0], arr[1], precision="fp64" if op == "fp64" else "mixed", max_sources=case["src"])
    if op == "grad":
        # the fit's parameters: gains, position and flux corrections to a catalogue
        cat = torch.from_numpy(_perturbed(case, seed, src)).cuda()
        return {"op": op, "p": p, "vis": vis, "cat": cat, "gain": gain64.requires_grad_(True),
                "dpos": torch.zeros((case["src"], 2), device="cuda", requires_grad=True),
                "dflux": torch.zeros((case["src"], 1), device="cuda", requires_grad=True)}
    if op == "predict":
        return {"op": op, "p": p, "src": src, "gain": gain64, "out": p.empty_cube()}
    if op == "fp64":
        vis = vis.to(torch.complex128)
    return {"op": op, "p": p, "src": src, "vis": vis, "resid": torch.empty_like(vis)}


def run(state):
    op = state["op"]
    if op == "grid":
        return state["g"].run(state["xy"], state["vis"], out=state["grid"])
    if op == "integrate":
        return state["g"].run(state["fine"], out=state["out"])
    if op == "solve":
        return state["p"].solve(state["avg"], state["S"])[0]
    if op == "predict":
        return state["p"].predict(state["src"], state["gain"], out=state["out"])
    if op == "grad":
        src = state["cat"] + torch.cat([state["dpos"], state["dflux"]], dim=1)
        loss = PeelLoss.apply(state["p"], state["vis"], state["gain"], src)
        g_gain, g_pos, g_flux = torch.autograd.grad(loss, (state["gain"], state["dpos"], state["dflux"]))
        # the loss is a sum of FP32 residuals: kept as such beside the gradients
        return {"loss": loss.detach().float(), "g_gain": g_gain, "g_pos": g_pos, "g_flux": g_flux}
    if op == "taylor":
        resid, gain, slope, _ = state["p"].cadence_taylor(state["vis"], state["src"], resid=state["resid"],
                                                          status=False)
        return {"resid": resid, "gain": gain, "slope": slope}
    # the streaming form: statuses are thresholds on the last change, read later if at all
    resid, jones, _ = state["p"].cadence(state["vis"], state["src"], resid=state["resid"], status=False)
    return {"resid": resid, "jones": jones}


# -- the same in 64 bits ----------------------------------------------------------

def _delays(arr, src_k):
    """[time][bl] delay in seconds and [time][bl] x 3 of what it is linear in."""
    uvw, _, ai, aj = arr
    u = torch.as_tensor(uvw, device="cuda")
    d = u[:, ai] - u[:, aj]
    return d @ _lmn(src_k[None])[:, 0] / C_LIGHT, d


def _phasor(arr, src_k):
    tau, _ = _delays(arr, src_k)
    turns = tau[..., None] * torch.as_tensor(arr[1], device="cuda")
    a = TAU * (turns - torch.round(turns))
    return torch.complex(torch.cos(a), -torch.sin(a))          # [time][bl][chan]


def _full(v, n_ant, ai, aj):
    """[ant][ant][2][2] of a Hermitian [bl][2][2], zero on the diagonal."""
    out = torch.zeros((n_ant, n_ant, 2, 2), dtype=torch.complex128, device="cuda")
    out[ai, aj] = v
    out[aj, ai] = _herm(v)
    return out


def _others(c):
    return c.sum(0, keepdim=True) - c


def _als(v, s, n_ant, arr, n_iter=20):
    v = _full(v, n_ant, arr[2], arr[3])
    j = torch.eye(2, dtype=torch.complex128, device="cuda").repeat(n_ant, 1, 1)
    for it in range(1, n_iter + 1):
        a = torch.einsum("pqab,qbc->pac", v, j) * s
        new = a @ torch.linalg.inv(_others(_herm(j) @ j) * s * s)
        j = 0.5 * (new + j) if it % 2 == 0 else new
    return j


def _als_taylor(mom, mu, s, n_ant, arr, n_iter=20):
    """Gains G + x H from the channel moments mom[n] = mean x^n R (n = 0, 1, 2) and
    mu[n] = mean x^n: Jacobi sweeps on [G H] with a Newton step along a common
    rotation H + i G K of the slopes after each sweep from the second."""
    full = [_full(m, n_ant, arr[2], arr[3]) for m in mom]
    eye = torch.eye(2, dtype=torch.complex128, device="cuda")
    g, h = eye.repeat(n_ant, 1, 1), torch.zeros((n_ant, 2, 2), dtype=torch.complex128, device="cuda")
    basis = torch.tensor([[[1, 0], [0, 0]], [[0, 0], [0, 1]], [[0, 1], [1, 0]], [[0, -1j], [1j, 0]]],
                         dtype=torch.complex128, device="cuda")
    both = basis[:, None] @ basis[None] + basis[None] @ basis[:, None]

    def mul(m, j):
        return torch.einsum("pqab,qbc->pac", m, j)

    for it in range(1, n_iter + 1):
        a = s * torch.cat([mul(full[0], g) + mul(full[1], h), mul(full[1], g) + mul(full[2], h)], dim=2)
        k0, k1, k2 = (_others(k) for k in (_herm(g) @ g, _herm(g) @ h + _herm(h) @ g, _herm(h) @ h))
        c = [mu[n] * k0 + mu[n + 1] * k1 + mu[n + 2] * k2 for n in range(3)]
        c = s * s * torch.cat([torch.cat([c[0], c[1]], dim=2), torch.cat([c[1], c[2]], dim=2)], dim=1)
        x = a @ torch.linalg.inv(c)
        gn, hn = x[:, :, :2], x[:, :, 2:]
        if it % 2 == 0:
            gn, hn = 0.5 * (gn + g), 0.5 * (hn + h)
        if it >= 2:
            gi, gj, hi, hj = gn[arr[2]], gn[arr[3]], hn[arr[2]], hn[arr[3]]
            rho = mom[2] - s * (mu[2] * gi @ _herm(gj) + mu[3] * (gi @ _herm(hj) + hi @ _herm(gj))
                                + mu[4] * hi @ _herm(hj))
            d = [1j * s * (gi @ b @ _herm(hj) - hi @ b @ _herm(gj)) for b in basis]
            grad = torch.stack([-2.0 * (rho.conj() * da).sum().real for da in d])
            hess = torch.stack([torch.stack([
                2.0 * mu[4] * (d[p].conj() * d[q]).sum().real
                - 2.0 * s * (rho.conj() * (gi @ both[p, q] @ _herm(gj))).sum().real for q in range(4)])
                for p in range(4)])
            low, info = torch.linalg.cholesky_ex(hess)
            if int(info) == 0 and bool((low.diagonal() ** 2).min() > 1e-6 * hess.diagonal().max()):
                step = torch.cholesky_solve(-grad[:, None], low)[:, 0]
                hn = hn + 1j * gn @ (step[:, None, None] * basis).sum(0)
        g, h = gn, hn
    return g, h


def _exact_peel(case, seed):
    arr, src, gain, slope, gen = _sky(case, seed)
    vis = _cube(case, arr, src, gain, slope, gen).to(torch.complex128)
    n_t, n_bl, n_c = vis.shape[:3]
    x = ((torch.arange(n_c, device="cuda", dtype=torch.float64) - (n_c - 1) / 2) / n_c)
    mu = [float((x ** n).mean()) for n in range(5)]
    gains, slopes = [], []
    for k in range(len(src)):
        e, s = _phasor(arr, src[k]), float(src[k, 2])
        if case["op"] == "taylor":
            z = torch.stack([torch.einsum("tbcp,tbc->bp", vis, e.conj() * x ** n) for n in range(3)])
            z = (z / (n_t * n_c)).reshape(3, n_bl, 2, 2)
            g, h = _als_taylor(z, mu, s, case["ant"], arr)
            slopes.append(h.reshape(-1, 4))
            gi, gj, hi, hj = g[arr[2]], g[arr[3]], h[arr[2]], h[arr[3]]
            m = [gi @ _herm(gj), gi @ _herm(hj) + hi @ _herm(gj), hi @ _herm(hj)]
        else:
            z = torch.einsum("tbcp,tbc->bp", vis, e.conj()) / (n_t * n_c)
            g = _als(z.reshape(n_bl, 2, 2), s, case["ant"], arr)
            m = [g[arr[2]] @ _herm(g[arr[3]])]
        gains.append(g.reshape(-1, 4))
        for n, mn in enumerate(m):
            vis -= s * mn.reshape(1, n_bl, 1, 4) * (e * x ** n)[..., None]
    if case["op"] == "taylor":
        return {"resid": vis, "gain": torch.stack(gains), "slope": torch.stack(slopes)}
    return {"resid": vis, "jones": torch.stack(gains)}


def _models(case, arr, src, jones):
    """Each source's 2x2 model [bl][4] before its phase."""
    for k in range(len(src)):
        yield float(src[k, 2]) * (jones[k][arr[2]] @ _herm(jones[k][arr[3]])).reshape(-1, 4)


def _exact_grad(case, seed):
    arr, src, gain, slope, gen = _sky(case, seed)
    r = _cube(case, arr, src, gain, slope, gen).to(torch.complex128)
    src = _perturbed(case, seed, src)
    gain = gain.to(torch.complex64).to(torch.complex128)
    for k, m in enumerate(_models(case, arr, src, gain)):
        r -= m[None, :, None, :] * _phasor(arr, src[k])[..., None]
    nu = torch.as_tensor(arr[1], device="cuda")
    g_gain = torch.zeros((case["src"], case["ant"], 2, 2), dtype=torch.complex128, device="cuda")
    g_pos, g_flux = [], []
    for k, m in enumerate(_models(case, arr, src, gain)):
        e, (_, d) = _phasor(arr, src[k]), _delays(arr, src[k])
        g0 = torch.einsum("tbcp,tbc->tbp", r, e.conj())
        g1 = torch.einsum("tbcp,tbc->tbp", r, e.conj() * nu)
        l, mm, s = (float(v) for v in src[k])
        n = math.sqrt(1.0 - l * l - mm * mm)
        # dL/dl = -2 Re sum conj(R) dV/dl, dV/dl = -2 pi i (nu / c) (u - w l / n) V
        w = (g1.conj() * m[None]).sum(-1).imag
        a = [d[..., 0] - d[..., 2] * (l / n), d[..., 1] - d[..., 2] * (mm / n)]
        g_pos.append(torch.stack([-2.0 * TAU / C_LIGHT * (w * ai).sum() for ai in a]))
        g = g0.sum(0)
        g_flux.append(-2.0 / s * (g.conj() * m).sum().real[None])
        g = g.reshape(-1, 2, 2)
        g_gain[k].index_add_(0, arr[2], -2.0 * s * g @ gain[k][arr[3]])
        g_gain[k].index_add_(0, arr[3], -2.0 * s * _herm(g) @ gain[k][arr[2]])
    return {"loss": (r.real ** 2).sum() + (r.imag ** 2).sum(), "g_gain": g_gain.reshape(case["src"], -1, 4),
            "g_pos": torch.stack(g_pos), "g_flux": torch.stack(g_flux)}


def _exact_predict(case, seed):
    arr, src, gain, _, _ = _sky(case, seed)
    gain = gain.to(torch.complex64).to(torch.complex128)
    out = torch.zeros((case["time"], arr[2].shape[0], case["chan"], 4), dtype=torch.complex128, device="cuda")
    for k, m in enumerate(_models(case, arr, src, gain)):
        out += m[None, :, None, :] * _phasor(arr, src[k])[..., None]
    return out


def _exact_grid(case, seed):
    xy, vis = _uv_points(case, seed)
    n, rmax = case["pix"], case["rmax"]
    inside = ((xy >= 0) & (xy < n)).all(dim=1)
    xy, vis = xy[inside].double(), vis[inside].to(torch.complex128)
    table = torch.as_tensor(_taper(), device="cuda")
    out = torch.zeros((case["pol"], n * n), dtype=torch.complex128, device="cuda")
    reach = int(math.ceil(rmax))
    base = torch.floor(xy)
    for dy in range(-reach, reach + 2):
        for dx in range(-reach, reach + 2):
            px, py = base[:, 0] + dx, base[:, 1] + dy
            r = torch.sqrt((px - xy[:, 0]) ** 2 + (py - xy[:, 1]) ** 2)
            ok = (r < rmax) & (px >= 0) & (px < n) & (py >= 0) & (py < n)
            at = r[ok] * ((len(table) - 1) / rmax)
            k = torch.clamp(at.long(), max=len(table) - 2)
            f = table[k] + (at - k) * (table[k + 1] - table[k])
            pix = (py[ok] * n + px[ok]).long()
            for pol in range(case["pol"]):
                v = f * vis[ok, pol]
                flat = torch.view_as_real(out[pol])
                flat[:, 0].index_add_(0, pix, v.real.contiguous())
                flat[:, 1].index_add_(0, pix, v.imag.contiguous())
    return out.reshape(case["pol"], n, n)


def _exact_integrate(case, seed):
    lengths, fine = _samples(case, seed)
    out = torch.zeros((4,) + tuple(fine.shape[1:]), dtype=torch.complex128, device="cuda")
    lengths = torch.as_tensor(lengths, device="cuda")
    for length in (16, 8, 4):
        rows = torch.nonzero(lengths == length)[:, 0]
        for slot in range(16 // length):
            mean = 0.0
            for t in range(slot * length, (slot + 1) * length):
                mean = mean + fine[t, rows].to(torch.complex128)
            out[slot, rows] = mean / length
    return out


def exact(case, seed):
    op = case["op"]
    if op == "grid":
        return _exact_grid(case, seed)
    if op == "integrate":
        return _exact_integrate(case, seed)
    if op == "solve":
        arr, src, avg = _averages(case, seed)
        return _als(avg.to(torch.complex128).reshape(-1, 2, 2), float(src[0, 2]), case["ant"], arr).reshape(-1, 4)
    n_vis = case["ant"] * (case["ant"] - 1) // 2 * case["chan"] * case["time"]
    if n_vis * case["src"] > 1e10:      # minutes at double precision
        return None
    if op == "grad":
        return _exact_grad(case, seed)
    if op == "predict":
        return _exact_predict(case, seed)
    return _exact_peel(case, seed)
