"""The work that a user of the engine has it do, as cases for timing.

Every case goes through the package's public entry points: ``Plan.search`` and
``Plan.search_stats`` (one segment of visibilities to candidates, and to every
image's statistics), ``Plan.render`` (images of listed trials),
``Plan.periodicity_search`` and ``rf_image_stats_noalloc``.  Sizes are those of
the repository's own workloads (``tiny``, ``realtime``, ``batching``, the
serving mix, the 4096^2 stress subset), with fewer DM trials where a whole
workload takes seconds, and ragged ones in between.

A state holds the visibilities (device memory, or page-locked host memory
where ``host`` is set) and the plan, which a program keeps from segment to
segment.  Visibilities are circular Gaussian noise of unit variance per
polarisation and one dispersed pulse some 15 sigma bright in its best image, so
that a search returns from a handful to a few hundred candidates.
"""

import math

import numpy as np
import torch

import paper_1802_03084_gb300 as rf

C_LIGHT = 299792458.0
K_DISP = 4.1488e-3                    # s GHz^2 per pc cm^-3
ARCSEC = math.pi / (180.0 * 3600.0)
PULSE_SNR = 15.0
LIST_SIZE = 2048

_SEARCH = dict(kind="search", nant=27, nchan=64, f_lo_ghz=1.0, bw_ghz=1.0, nint=128, tint_ms=5.0, npol=2, npix=256,
               cell_arcsec=10.0, ndm=8, dm_max=700.0, dm_grid="linear", dts="1", threshold=7.0, fp16=False,
               partial=False, mean_subtract=False, clipped=False, host=False, continuum=0.0)


def _case(**kw):
    return dict(_SEARCH, **kw)


def listed():
    return [
        # the smallest calls: one uv half plane imaged inside a caller's own
        # loop or graph, where launches and latency are all there is
        dict(name="halfplane_256", kind="noalloc", npix=256),
        dict(name="halfplane_1024", kind="noalloc", npix=1024),
        # the smallest segment search (the `tiny` workload), every image's
        # statistics returned, partial sweeps searched
        _case(name="tiny_stats", kind="stats", partial=True, threshold=6.0),
        # a short segment of the serving mix, read from pinned host memory
        _case(name="serving_512_host", nchan=64, nint=512, npix=512, ndm=60, dm_max=1500.0, dm_grid="smearing",
              dts="1,2,4", host=True),
        # ragged sizes, one polarisation, widths that do not divide each other
        _case(name="ragged_512_stats", kind="stats", nant=21, nchan=100, nint=333, npol=1, npix=512, ndm=7,
              dm_max=400.0, dts="1,3,5", threshold=6.5),
        # steady sources removed, noise from the clipped pixels
        _case(name="clipped_512", nchan=128, nint=512, npix=512, ndm=32, dm_max=800.0, dm_grid="smearing",
              dts="1,2,4", mean_subtract=True, clipped=True, continuum=0.02),
        # the `realtime` workload: one whole segment
        _case(name="realtime_1024", nchan=256, nint=1024, npix=1024, ndm=128, dm_max=1500.0, dm_grid="smearing",
              dts="1,2,4,8"),
        # the `batching` workload (FP16 storage) with one DM trial in eight
        _case(name="batching_2048", nchan=1024, nint=2048, npix=2048, ndm=32, dm_max=3000.0, dts="1,2,4,8,16",
              fp16=True),
        # the 4096^2 stress subset: 64 integrations around a pulse, strong
        # steady source, FP16 storage
        _case(name="stress_4096", nchan=2048, bw_ghz=2.0, nint=64, tint_ms=10.0, npix=4096, ndm=4, dm_max=300.0,
              dts="1,2,4,8,16,32", fp16=True, partial=True, continuum=50.0),
        # periodic signals: every fluctuation frequency of a window imaged
        _case(name="periodic_1024", kind="periodic", nchan=256, nint=1024, npix=1024, ndm=32, dm_max=600.0,
              L=128, kmin=1, kmax=64),
        # images of the candidates of a segment, for their plots
        _case(name="render_1024", kind="render", nchan=256, nint=1024, npix=1024, ndm=32, dm_max=600.0,
              dts="1,2,4,8", nimages=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a search of any size, or one of the other calls."""
    most = _cost(next(c for c in listed() if c["name"] == "batching_2048"))
    while True:
        kind = rng.choice(["search", "search", "search", "stats", "noalloc", "periodic", "render"])
        if kind == "noalloc":
            return dict(kind=kind, npix=rng.choice([64, 128, 512, 1024]), occupied=rng.uniform(0.01, 0.3))
        npix = rng.choice([512, 1024, 2048, 4096] if kind == "stats" else [256, 512, 1024, 2048])
        nint = _log(rng, 64, 1500)
        c = _case(kind=kind, npix=npix, nint=nint, nchan=_log(rng, 16, 700), nant=rng.choice([18, 21, 24, 27]),
                  npol=rng.choice([1, 2, 2]), tint_ms=rng.choice([2.0, 5.0, 10.0]), ndm=_log(rng, 2, 40),
                  dm_max=rng.uniform(50.0, 900.0), dm_grid=rng.choice(["linear", "smearing"]),
                  dts=rng.choice(["1", "1,2", "1,2,4", "1,2,4,8", "1,2,4,8,16", "1,2,3,4,6", "2,4,8", "1,4,16", "1,3,9"]),
                  fp16=rng.random() < 0.4, partial=rng.random() < 0.4, mean_subtract=rng.random() < 0.2,
                  clipped=kind == "search" and rng.random() < 0.2, host=rng.random() < 0.15,
                  threshold=rng.choice([6.5, 7.0]))
        if kind == "periodic":
            L = 1 << rng.randint(4, 8)
            kmin = rng.randint(1, 3)
            c.update(L=L, kmin=kmin, kmax=rng.randint(kmin + 1, min(L // 2, 64)), dts="1", dm_max=c["dm_max"] / 4)
            if L + _delays(c).max() > nint:
                continue
        if kind == "render":
            c.update(nimages=rng.randint(1, 12))
        n = _count(c)
        if n < 4 or (kind == "stats" and n > 4000) or _cost(c) > most:
            continue
        return c


# ------------------------------------------------------------ plan geometry
def _dts(c):
    return [int(x) for x in c["dts"].split(",")]


def _freqs(c):
    return (c["f_lo_ghz"] + (np.arange(c["nchan"]) + 0.5) * (c["bw_ghz"] / c["nchan"])) * 1e9


def _antennas(c):
    """A Y of three arms, log-spaced radii 40 .. 600 m, hour angle 0, declination +30."""
    per, rng = c["nant"] // 3, np.random.default_rng(c["nant"])
    radii, pos = np.geomspace(40.0, 600.0, per), []
    for arm in range(3):
        r = radii * np.append(rng.uniform(0.95, 1.0, per - 1), 1.0)
        az = 0.31 + arm * 2.0 * math.pi / 3.0
        pos.append(np.stack([r * math.sin(az), r * math.cos(az) * math.cos(math.radians(4.0784)),
                             -r * math.cos(az) * math.sin(math.radians(4.0784))], axis=1))
    return np.concatenate(pos)


def _baselines(c):
    a = _antennas(c)
    i, j = np.triu_indices(c["nant"], k=1)
    return a[j] - a[i]


def _dms(c):
    if c["dm_grid"] == "linear":
        return np.linspace(0.0, c["dm_max"], c["ndm"])
    # equal steps of one effective pulse width of added delay
    a = 2.0 * K_DISP * (c["bw_ghz"] / c["nchan"]) / (_freqs(c).min() * 1e-9) ** 3
    tint = c["tint_ms"] * 1e-3
    return (tint / a) * np.sinh(np.linspace(0.0, 1.0, c["ndm"]) * math.asinh(a * c["dm_max"] / tint))


def _delays(c):
    f = _freqs(c) * 1e-9
    x = (K_DISP * _dms(c))[:, None] * (1.0 / (f * f) - 1.0 / (f.max() * f.max()))[None, :]
    return np.floor(x / (c["tint_ms"] * 1e-3) + 0.5).astype(np.int64)


def _times(c):
    """Images per (DM, dt)."""
    mx, n = _delays(c).max(axis=1), c["nint"]
    return [[n // dt if c["partial"] else max(n - int(m), 0) // dt for dt in _dts(c)] for m in mx]


def _count(c):
    if c["kind"] == "periodic":
        return 2 * int((_delays(c).max(axis=1) + c["L"] <= c["nint"]).sum()) * (c["kmax"] - c["kmin"] + 1)
    if c["kind"] == "render":
        return min(c["nimages"], sum(map(sum, _times(c))))
    return sum(map(sum, _times(c)))


def _fft_flops(n, ncol):
    """One image from its half plane: ncol column transforms, one complex row transform per two rows."""
    return (ncol + n // 2) * 5.0 * n * math.log2(n)


def _columns(c):
    fov = c["npix"] * c["cell_arcsec"] * ARCSEC
    return min(int(np.abs(_baselines(c)[:, 0]).max() * _freqs(c).max() / C_LIGHT * fov) + 2, c["npix"] // 2)


def _cost(c):
    n = c["npix"]
    return _count(c) * _fft_flops(n, n // 3) + 50.0 * c["nint"] * c["nchan"] * c["nant"] ** 2


def work(case):
    n = case["npix"]
    if case["kind"] == "noalloc":
        return {"bytes": n * (n // 2 + 1) * 8 + 48, "flops": _fft_flops(n, n // 2)}
    nvis = case["nant"] * (case["nant"] - 1) // 2 * case["nchan"]
    vis = case["nint"] * nvis * case["npol"] * 8
    fft = _fft_flops(n, _columns(case))
    images = _count(case)
    if case["kind"] == "render":
        return {"bytes": vis + images * n * n * 4, "flops": images * (fft + 2.0 * nvis)}
    if case["kind"] == "periodic":
        return {"bytes": vis + images // 2 * 64, "flops": images * (fft + 2.0 * nvis + 2.0 * n * n)}
    # an image of a width that another width of the list divides is the sum of
    # that width's images: the transforms are those of the other widths only
    dts = _dts(case)
    own = [k for k, dt in enumerate(dts) if not any(dt % o == 0 for o in dts if o < dt)]
    made = sum(row[k] for row in _times(case) for k in own)
    return {"bytes": vis + images * (56 if case["kind"] == "stats" else 0),
            "flops": made * (fft + 2.0 * nvis) + images * 2.0 * n * n}


# ------------------------------------------------------------------- inputs
def _phases(c, x, y):
    bl, f = _baselines(c), _freqs(c)
    cell = c["cell_arcsec"] * ARCSEC
    lm = ((x - c["npix"] // 2) * cell, (y - c["npix"] // 2) * cell)
    return np.exp(-2j * math.pi * np.outer(bl[:, 0] * lm[0] + bl[:, 1] * lm[1], f / C_LIGHT))


def _visibilities(c, seed):
    nbl, nchan, nint, npol = c["nant"] * (c["nant"] - 1) // 2, c["nchan"], c["nint"], c["npol"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    vis = torch.empty((nint, nbl, nchan, npol), dtype=torch.complex64, device="cuda")
    step = max(1, (1 << 27) // (nbl * nchan * npol))
    for t in range(0, nint, step):  # E|n|^2 = 1 per polarisation
        vis[t:t + step] = torch.randn(vis[t:t + step].shape, dtype=torch.complex64, device="cuda", generator=g)
    r = np.random.default_rng(seed)
    n, span = c["npix"], c["npix"] // 8
    if c["continuum"]:
        vis += torch.from_numpy((c["continuum"] * _phases(c, n // 2 + span // 3, n // 2 - span // 2))
                                .astype(np.complex64)).cuda()[None, :, :, None]
    # one pulse of two integrations at a trial DM whose sweep fits the segment
    dms, sweep = _dms(c), _delays(c).max(axis=1)
    fit = np.nonzero(sweep + 4 < nint)[0]
    d = int(fit[r.integers((len(fit) + 1) // 2, len(fit) + 1) - 1])
    x, y = (int(v) for v in r.integers(n // 2 - span, n // 2 + span, 2))
    f, tint = _freqs(c) * 1e-9, c["tint_ms"] * 1e-3
    start = r.uniform(0.0, nint - 3.0 - sweep[d]) + K_DISP * dms[d] * (f ** -2 - f.max() ** -2) / tint
    amp = PULSE_SNR * 0.5 * math.sqrt(2.0 / npol) / math.sqrt(2.0 * nbl * nchan)
    ph = torch.from_numpy((amp * _phases(c, x, y)).astype(np.complex64)).cuda()
    first = np.floor(start).astype(np.int64)
    for k in range(3):
        t = first + k
        share = np.clip(np.minimum(start + 2.0, t + 1) - np.maximum(start, t), 0.0, 1.0)
        ok = np.nonzero((t >= 0) & (t < nint) & (share > 0))[0]
        tt, cc = torch.from_numpy(t[ok]).cuda(), torch.from_numpy(ok).cuda()
        add = ph[:, cc].T * torch.from_numpy(share[ok].astype(np.float32)).cuda()[:, None]
        vis[tt, :, cc, :] += add[:, :, None]
    if c["kind"] == "periodic":  # a source that varies at one of the imaged frequencies
        k = (c["kmin"] + c["kmax"]) // 2
        wave = torch.cos(2 * math.pi * k / c["L"] * torch.arange(nint, device="cuda", dtype=torch.float64)).float()
        vis += (3.0 * wave / math.sqrt(c["L"]))[:, None, None, None] * ph[None, :, :, None]
    return vis


def _half_plane(c, seed):
    """A uv half plane with a share of its cells occupied, column 0 Hermitian, column N/2 empty."""
    n = c["npix"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    h = torch.randn((n, n // 2 + 1), dtype=torch.complex64, device="cuda", generator=g)
    h *= torch.rand((n, n // 2 + 1), device="cuda", generator=g) < c.get("occupied", 0.05)
    h[:, -1] = 0
    h[n // 2, :] = 0
    flip = (-torch.arange(n, device="cuda")) % n
    h[:, 0] = h[:, 0] + h[flip, 0].conj()
    return h, float(max(int((h != 0).sum()), 1))


def _trials(c, seed):
    times = _times(c)
    every = [(d, s) for d, row in enumerate(times) for s, n in enumerate(row) if n > 0]
    r = np.random.default_rng(seed + 1)
    return sorted({(d, s, int(r.integers(times[d][s]))) for d, s in (every[i] for i in r.integers(0, len(every), _count(c)))})


def prepare(case, seed):
    if case["kind"] == "noalloc":
        h, w = _half_plane(case, seed)
        return {"case": case, "half": h, "weight": w, "stat": torch.zeros(6, dtype=torch.float64, device="cuda")}
    vis = _visibilities(case, seed)
    flags = (rf.RF_STORE_FP16 * case["fp16"] | rf.RF_EDGE_PARTIAL * case["partial"] |
             rf.RF_MEAN_SUBTRACT * case["mean_subtract"] | rf.RF_NOISE_CLIPPED * case["clipped"])
    plan = rf.Plan(_antennas(case), _freqs(case), case["tint_ms"] * 1e-3, case["npix"], case["cell_arcsec"] * ARCSEC,
                   _dms(case), _dts(case), case["threshold"], npol=case["npol"], flags=flags, max_nint=case["nint"])
    if case["host"]:
        vis = vis.cpu().pin_memory()
    s = {"case": case, "vis": vis, "plan": plan}
    if case["kind"] == "render":
        s["trials"] = _trials(case, seed)
    return s


# ---------------------------------------------------------------- the calls
def _columns_of(a):
    return {k: np.ascontiguousarray(a[k]) for k in a.dtype.names if k != "pad"}


def _list_of(a):
    """A candidate list of any length as its length and columns of a fixed one (a caller's fixed-size record)."""
    size = max(LIST_SIZE, len(a))
    return dict({k: np.concatenate([v, np.zeros(size - len(a), v.dtype)]) for k, v in _columns_of(a).items()},
                found=len(a))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "noalloc":
        stat = state["stat"]
        rf.rf_image_stats_noalloc(state["half"], case["npix"], state["weight"], stat)
        return {"index": stat.view(torch.int32)[:5], "peak_sigma_snr": stat.view(torch.float32)[5:8],
                "mean_weight": stat[4:6]}
    plan, vis = state["plan"], state["vis"]
    if kind == "search":
        return _list_of(plan.search(vis))
    if kind == "stats":
        cands, stats = plan.search_stats(vis)
        return {"candidates": _list_of(cands), "images": _columns_of(stats)}
    if kind == "periodic":
        cands, stats = plan.periodicity_search(vis, case["L"], case["kmin"], case["kmax"], case["threshold"],
                                               with_stats=True)
        return {"candidates": _list_of(cands), "images": _columns_of(stats)}
    return plan.render(vis, state["trials"])


# -------------------------------------------------- the same in 64 bits
def _cells(c):
    fov = c["npix"] * (c["cell_arcsec"] * ARCSEC)
    s = _freqs(c) / C_LIGHT
    bl, half = _baselines(c), c["npix"] // 2
    iu, iv = (np.sign(x) * np.floor(np.abs(x) + 0.5) for x in ((bl[:, 0][:, None] * s) * fov, (bl[:, 1][:, None] * s) * fov))
    on = (np.abs(iu) < half) & (np.abs(iv) < half)
    return iu.astype(np.int64), iv.astype(np.int64), on


class _Imager:
    """Dirty images of [n][nbl][nchan] visibilities: every on-grid one and its mirror, nearest cell."""

    def __init__(self, c):
        self.n = n = c["npix"]
        iu, iv, on = _cells(c)
        self.on = torch.from_numpy(on).cuda()
        u, v = iu[on], iv[on]
        self.at = torch.from_numpy(np.concatenate([(v % n) * n + u % n, (-v % n) * n + (-u) % n])).cuda()
        self.sign = torch.from_numpy(np.where((u + v) % 2, -1.0, 1.0)).cuda()
        self.per_chan = torch.from_numpy(on.sum(axis=0)).cuda()

    def __call__(self, R, W):
        r = R[:, self.on] * self.sign
        g = torch.zeros((R.shape[0], self.n * self.n), dtype=torch.complex128, device="cuda")
        g.index_add_(1, self.at, torch.cat([r, r.conj()], dim=1))
        img = torch.fft.ifft2(g.view(-1, self.n, self.n)).real * (self.n * self.n)
        return img / (2.0 * W[:, None, None])


def _padded(v):
    return np.concatenate([v, np.zeros(max(LIST_SIZE - len(v), 0))])


def _stored(c, S):
    """The stored samples: rounded to FP16 where the plan's caller chose that."""
    if c["fp16"]:
        S = torch.view_as_complex(torch.view_as_real(S).float().half().double())
    return S


def _stokes(c, vis):
    out = torch.empty(vis.shape[:3], dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 26) // vis[0].numel())
    for t in range(0, len(vis), step):
        out[t:t + step] = vis[t:t + step].cuda().to(torch.complex128).mean(dim=3)
    out = _stored(c, out)
    if c["mean_subtract"]:
        out = _stored(c, out - out.mean(dim=0, keepdim=True))
    return out


def _samples(c, S, delay, dt, t):
    """Boxcar sums of dt samples after the delay at output times t, and the samples in each per channel."""
    nint, chan = len(S), torch.arange(S.shape[2], device="cuda")
    delay = torch.from_numpy(delay).cuda()
    R = torch.zeros((len(t),) + S.shape[1:], dtype=torch.complex128, device="cuda")
    have = torch.zeros((len(t), S.shape[2]), dtype=torch.float64, device="cuda")
    for j in range(dt):
        at = t[:, None] * dt + j + delay[None, :]
        ok = at < nint
        # advanced indexes around a slice: [time][channel][baseline]
        R += (S[at.clamp(max=nint - 1), :, chan] * ok[:, :, None]).transpose(1, 2)
        have += ok
    return R, have


def _image_stats(c, img):
    n = img.shape[-1]
    flat = img.reshape(len(img), -1)
    peak, at = flat.max(dim=1)
    mean = flat.mean(dim=1)
    sigma = (flat - mean[:, None]).square().mean(dim=1).sqrt()
    if c["clipped"]:
        keep = (flat - mean[:, None]).abs() <= 5.0 * sigma[:, None]
        count = keep.sum(dim=1)
        mean = (flat * keep).sum(dim=1) / count
        sigma = (((flat - mean[:, None]) * keep).square().sum(dim=1) / count).sqrt()
    return peak, sigma, mean, at % n, at // n


def exact(case, seed):
    n = case["npix"]
    if case["kind"] == "noalloc":
        h, w = _half_plane(case, seed)
        h = h.to(torch.complex128)
        g = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
        flip = (-torch.arange(n, device="cuda")) % n
        g[:, :n // 2] = h[:, :n // 2]
        g[:, n // 2 + 1:] = h[flip][:, 1:n // 2].conj().flip(1)
        par = torch.arange(n, device="cuda") % 2
        g = torch.where((par[:, None] + par[None, :]) % 2 == 1, -g, g)
        img = torch.fft.ifft2(g).real * (n * n) / (2.0 * w)
        peak, sigma, mean, x, y = _image_stats({"clipped": False}, img[None])
        return {"index": None, "peak_sigma_snr": torch.cat([peak, sigma, peak / sigma]),
                "mean_weight": None}
    if _count(case) * n * n > 1e10 or case["nint"] * case["nchan"] * case["nant"] ** 2 > (1 << 28):
        return None
    vis = _visibilities(case, seed)
    S = _stokes(case, vis)
    del vis
    imager, delays, dts = _Imager(case), _delays(case), _dts(case)
    batch = max(1, min(64, (1 << 27) // max(n * n, S[0].numel())))
    if case["kind"] == "render":
        out = np.empty((0, n, n))
        for d, s, t in _trials(case, seed):
            R, have = _samples(case, S, delays[d], dts[s], torch.tensor([t], device="cuda"))
            out = np.concatenate([out, imager(R, (have * imager.per_chan).sum(dim=1)).cpu().numpy()])
        return out
    if case["kind"] == "periodic":
        return _exact_periodic(case, S, imager, delays, batch)
    cols = {k: [] for k in ("dm_idx", "dt_idx", "t_idx", "x", "y", "peak", "sigma", "snr", "mean", "weight")}
    for d, row in enumerate(_times(case)):
        for s, nt in enumerate(row):
            for t0 in range(0, nt, batch):
                t = torch.arange(t0, min(nt, t0 + batch), device="cuda")
                R, have = _samples(case, S, delays[d], dts[s], t)
                W = (have * imager.per_chan).sum(dim=1)
                peak, sigma, mean, x, y = _image_stats(case, imager(R, W))
                same = torch.full_like(t, 1)
                for k, v in zip(cols, (same * d, same * s, t, x, y, peak, sigma, peak / sigma, mean, W)):
                    cols[k].append(v.cpu().numpy())
    a = {k: np.concatenate(v) for k, v in cols.items()}
    found = a["snr"] >= case["threshold"]
    cands = {k: _padded(a[k][found]) for k in ("snr", "peak", "sigma")}
    if case["kind"] == "stats":
        return {"candidates": cands, "images": {k: a[k] for k in ("peak", "sigma", "snr", "weight")}}
    return cands


def _exact_periodic(c, S, imager, delays, batch):
    L, n = c["L"], c["npix"]
    ks = torch.arange(c["kmin"], c["kmax"] + 1, device="cuda")
    turn = 2.0 * math.pi / L * ((ks[:, None] * torch.arange(L, device="cuda")[None, :]) % L).double()
    amp, sig = [], []
    for row in delays:
        if row.max() + L > c["nint"]:
            continue
        x = _samples(c, S, row, 1, torch.arange(L, device="cuda"))[0].reshape(L, -1)
        U, Q = ((f(turn).to(torch.complex128) @ x / L).reshape((-1,) + S.shape[1:]) for f in (torch.cos, torch.sin))
        for k in range(0, len(ks), batch):
            W = imager.per_chan.sum().double().expand(len(ks[k:k + batch]))
            iu, iq = imager(U[k:k + batch], W), imager(Q[k:k + batch], W)
            amp.append((iu.square() + iq.square()).flatten(1).amax(dim=1).sqrt().cpu().numpy())
            sig.append(((iu.flatten(1).var(dim=1, correction=0) + iq.flatten(1).var(dim=1, correction=0)) / 2).sqrt().cpu().numpy())
    amp, sig = np.concatenate(amp), np.concatenate(sig)
    found = amp / sig >= c["threshold"]
    return {"candidates": {"snr": _padded((amp / sig)[found]), "amplitude": _padded(amp[found]),
                           "sigma": _padded(sig[found])},
            "images": {"snr": amp / sig, "amplitude": amp, "sigma": sig}}
