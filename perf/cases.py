"""The workloads that the library's speed is judged on: what a user's program has it do, through
its public entry points, from one small lat-lon map to a mixed-resolution batch at nside 4096.

listed() names them, draw() gives others of the same ranges, prepare() makes what a program has
in hand before the call (grid, kernels, maps, buffers), run() is one pass, work() the bytes and
operations a pass cannot do without and exact() its result in 64 bits, restated here with plain
torch: ring DFTs, the sampled kernel's ring-pair coefficients, the band sum and the synthesis.

A case is a dict of plain values:
  op       "convolve" (maps on the GPU), "fit" (forward and backward: gradients of the maps and
           of the profile's knots), "multi" (several kernels on the same maps, summed with
           weights), "batch" (maps of several resolutions in one call), "host" (maps in pinned
           host memory, result back in pinned host memory)
  grid     "healpix" (nside) or "ecp" (ntheta x nphi)
  maps     maps per call;  beams: distinct kernels (1, or one per map, or the kernels of multi)
  profile  "gaussian" (fwhm, spread relatively over the beams by `spread`) or "mexican_hat"
  support  radius of the kernel; fwhm and support in arcminutes;  knots: of the tabulated profile
  form     "tf32" (3xTF32 tensor-core form) or "fp32" (plain form);  basic: the BASIC variant
"""
import math

import numpy as np
import torch

import paper_1104_0672_gb300 as ark
from paper_1104_0672_gb300 import inputs

ARCMIN = math.pi / (180.0 * 60.0)


def _case(name=None, op="convolve", grid="healpix", nside=0, ntheta=0, nphi=0, maps=1, beams=1, profile="gaussian",
          fwhm=5.0, spread=0.0, support=15.0, knots=256, form="tf32", basic=False, buffers=False, **more):
    c = dict(op=op, grid=grid, nside=nside, ntheta=ntheta, nphi=nphi, maps=maps, beams=beams, profile=profile,
             fwhm=fwhm, spread=spread, support=support, knots=knots, form=form, basic=basic, buffers=buffers, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one coarse lat-lon map and a wide Gaussian: the smallest call, launches and host work
        _case("ecp128_single", grid="ecp", ntheta=128, nphi=256, fwhm=240.0, support=720.0, form="fp32"),
        # a quarter-degree lat-lon grid with the odd ring count and the non-power-of-two ring
        # length of real ones, three fields
        _case("ecp721x1440_3maps", grid="ecp", ntheta=721, nphi=1440, maps=3, fwhm=60.0, support=180.0),
        # a single low-resolution sky map smoothed to 40', as before a component separation
        _case("hp256_single", nside=256, fwhm=40.0, support=120.0, form="fp32"),
        # a few medium maps, in the BASIC variant
        _case("hp512_basic_4maps", nside=512, maps=4, fwhm=20.0, support=60.0, basic=True),
        # many detector maps, each with its own beam
        _case("hp1024_64beams", nside=1024, maps=64, beams=64, fwhm=7.25, spread=0.38, support=0.0, buffers=True),
        # the benchmark's step: a batch of full-resolution maps with one shared 5' beam
        _case("hp2048_16maps", nside=2048, maps=16, buffers=True),
        # beam fitting at full resolution: forward and both gradients of one map
        _case("fit_hp2048", op="fit", nside=2048),
        # beam fitting of four detectors at low resolution, plain FP32 form
        _case("fit_hp256_4beams", op="fit", nside=256, maps=4, beams=4, fwhm=40.0, spread=0.1, support=120.0,
              form="fp32"),
        # an asymmetric beam as the weighted sum of ten symmetric ones
        _case("multi10_hp2048", op="multi", nside=2048, beams=10, fwhm=4.86, spread=0.074, support=0.0),
        # the paper's support of a degree at full resolution: over 32 input rings per output ring
        _case("wide_hp2048", nside=2048, fwhm=20.0, support=60.0),
        # fine-scale wavelet filtering of 16 maps of three resolutions in one call
        _case("wavelet_mixed_16maps", op="batch", nside=4096, maps=6, nside2=2048, maps2=5, nside3=512, maps3=5,
              profile="mexican_hat", fwhm=2.0, support=8.0, form="fp32", buffers=True),
        # maps that live on the host: copies and convolutions in a pipeline of two-map chunks
        _case("host_hp1024_8maps", op="host", nside=1024, maps=8, fwhm=10.0, support=30.0, buffers=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the ranges above: any resolution up to the listed ones (half of them powers
    of two, as sky maps mostly are), supports from a few rings to far over the 32 of the narrow
    path, one to many maps."""
    kind = rng.choice(["hp", "hp", "hp", "ecp", "fit", "multi", "wide", "batch", "host"])
    form = rng.choice(["tf32", "tf32", "fp32"])
    knots = rng.choice([64, 129, 256, 256, 500])

    def nside(lo, hi):
        n = _log_int(rng, lo, hi)
        return 1 << max(0, round(math.log2(n))) if rng.random() < 0.5 else n

    def rings(ns, r):  # support of about r input rings, in arcminutes
        return r * math.sqrt(math.pi / 3.0) / (2.0 * 1.4 * ns) / ARCMIN

    if kind == "ecp":
        nt = _log_int(rng, 48, 1024)
        s = rng.uniform(4.0, 15.0) * 180.0 * 60.0 / nt
        return _case(grid="ecp", ntheta=nt, nphi=2 * (nt + rng.randrange(-8, 9)), maps=rng.randrange(1, 9),
                     fwhm=s / 3.0, support=s, knots=knots, form=form)
    if kind == "wide":
        ns = nside(64, 1024)
        s = min(rings(ns, rng.uniform(36.0, 100.0)), 2400.0)
        return _case(nside=ns, maps=rng.randrange(1, 3), fwhm=s / 3.0, support=s, knots=knots, form=form)
    if kind == "batch":
        n1 = nside(128, 2048)
        s = rings(n1, rng.uniform(8.0, 24.0))
        return _case(op="batch", nside=n1, maps=rng.randrange(1, 4), nside2=max(16, n1 // 2), maps2=rng.randrange(1, 5),
                     nside3=max(8, n1 // 4 + 1), maps3=rng.randrange(1, 5), profile="mexican_hat", fwhm=s / 4.0,
                     support=s, knots=knots, form=form, buffers=True)
    top = {"hp": 2048, "fit": 1024, "multi": 1024, "host": 512}[kind]
    ns = nside({"host": 64}.get(kind, 16), top)
    s = min(rings(ns, rng.uniform(6.0, 26.0)), 2400.0)
    many = max(1, min(24, int(4.0e8 / (12 * ns * ns)) // 2))
    if kind == "multi":
        k = rng.randrange(2, 13)
        return _case(op="multi", nside=ns, maps=rng.randrange(1, 3), beams=k, fwhm=s / 3.6, spread=0.2, support=0.0,
                     knots=knots, form=form)
    maps = rng.randrange(1, many + 1)
    if kind == "host":
        return _case(op="host", nside=ns, maps=min(maps, 8), fwhm=s / 3.0, support=s, knots=knots, form=form,
                     buffers=True)
    if kind == "fit":
        maps = min(maps, 4)
    own = rng.random() < 0.35
    return _case(op="fit" if kind == "fit" else "convolve", nside=ns, maps=maps, beams=maps if own else 1,
                 fwhm=s / (3.6 if own else 3.0), spread=0.2 if own else 0.0, support=0.0 if own else s, knots=knots,
                 form=form, basic=kind == "hp" and rng.random() < 0.2, buffers=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
def _grids(case):
    """[(kind, sizes..., maps)] of a case, one entry but for "batch"."""
    if case["grid"] == "ecp":
        return [("ecp", case["ntheta"], case["nphi"], case["maps"])]
    g = [("healpix", case["nside"], 0, case["maps"])]
    for k in ("2", "3"):
        if case["op"] == "batch":
            g.append(("healpix", case["nside" + k], 0, case["maps" + k]))
    return g


def _profiles(case):
    """[(knots, support radius)] of the case's kernels.  support 0: three FWHM of each beam."""
    out = []
    nb = case["beams"]
    for b in range(nb):
        f = case["fwhm"] * (1.0 + case["spread"] * (2.0 * b / (nb - 1) - 1.0 if nb > 1 else 0.0)) * ARCMIN
        g = case["support"] * ARCMIN if case["support"] > 0 else 3.0 * f
        make = inputs.mexican_hat_knots if case["profile"] == "mexican_hat" else inputs.gaussian_knots
        k = make(f, g, case["knots"])
        if case["op"] == "fit":  # a fitted profile is a float32 parameter, of unit scale, that training has moved
            t = np.arange(case["knots"], dtype=np.float64)
            k = (k / np.abs(k).max() * (1.0 + 0.01 * np.sin(0.37 * t + b))).astype(np.float32).astype(np.float64)
        out.append((k, g))
    return out


def _weights(case, seed):
    return np.random.Generator(np.random.PCG64(int(seed))).uniform(-0.3, 1.0, case["beams"])


def _npix(g):
    return g[1] * g[2] if g[0] == "ecp" else 12 * g[1] * g[1]


def _maps(case, seed, device):
    """White-noise maps of every grid (and output gradients for "fit"), from the seed alone."""
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed) + 11040672)
    maps = [torch.randn((g[3], _npix(g)), generator=gen, dtype=torch.float32, device=device) for g in _grids(case)]
    grad = [torch.randn(m.shape, generator=gen, dtype=torch.float32, device=device) for m in maps] if case["op"] == "fit" else []
    return maps, grad


def _flags(case):
    return (ark.FLAG_3XTF32 if case["form"] == "tf32" else 0) | (ark.FLAG_BASIC if case["basic"] else 0)


def prepare(case, seed):
    dev = torch.device("cuda")
    maps, grad = _maps(case, seed, dev)
    grids = [ark.Grid.ecp(g[1], g[2]) if g[0] == "ecp" else ark.Grid.healpix(g[1]) for g in _grids(case)]
    prof = _profiles(case)
    kernels = [[ark.Kernel(g, k, gm) for k, gm in prof] for g in grids]
    kernels = [k[0] if len(k) == 1 else k for k in kernels]
    s = dict(case=case, flags=_flags(case), grids=grids, kernels=kernels, maps=maps, out=None, ws=None)
    op = case["op"]
    if op == "fit":
        s["maps"] = [maps[0].requires_grad_(True)]
        s["grad"] = grad[0]
        s["knots"] = torch.tensor(np.stack([k for k, _ in prof]), dtype=torch.float32, device=dev).requires_grad_(True)
    elif op == "multi":
        s["weights"] = _weights(case, seed)
    elif op == "batch":
        s["jobs"] = [(g, k, m, s["flags"]) for g, k, m in zip(grids, kernels, maps)]
        s["ws"] = torch.empty(ark.batch_workspace_size(s["jobs"]), dtype=torch.uint8, device=dev)
    elif op == "host":
        s["maps"] = [maps[0].cpu().pin_memory()]
        s["out"] = torch.empty_like(s["maps"][0]).pin_memory()
        s["ws"] = torch.empty(ark.host_workspace_size(grids[0], kernels[0], case["maps"], 2, s["flags"]),
                              dtype=torch.uint8, device=dev)
    elif case["buffers"]:  # a loop over batches keeps its output and workspace
        s["out"] = torch.empty_like(maps[0])
        s["ws"] = torch.empty(ark.workspace_size(grids[0], kernels[0], case["maps"], s["flags"]), dtype=torch.uint8,
                              device=dev)
    return s


def run(state):
    s, op = state, state["case"]["op"]
    g, k, x = s["grids"][0], s["kernels"][0], s["maps"][0]
    if op == "fit":
        y = ark.convolve_autograd(g, k, x, s["knots"].double(), s["flags"])
        return (y.detach(), *torch.autograd.grad(y, [x, s["knots"]], s["grad"]))
    if op == "multi":
        return ark.convolve_multi(g, k, x, weights=s["weights"], flags=s["flags"])
    if op == "batch":
        return ark.convolve_batch(s["jobs"], workspace=s["ws"])
    if op == "host":
        return ark.convolve_host(g, k, x, flags=s["flags"], out=s["out"], maps_per_chunk=2, workspace=s["ws"])
    return ark.convolve(g, k, x, flags=s["flags"], out=s["out"], workspace=s["ws"])


# ------------------------------------------------------------------ the operator's geometry
def _rings(g):
    """Per ring: colatitude, pixels, first-pixel longitude, pixel weight; and the kernel grid N."""
    if g[0] == "ecp":
        nt, nphi = g[1], g[2]
        th = (np.arange(nt) + 0.5) * math.pi / nt
        k = np.arange(1, nt // 2 + 1, dtype=np.float64)
        s = np.array([np.sum(np.cos(2.0 * k * t) / (4.0 * k * k - 1.0)) for t in th])
        w = (2.0 / nt) * (1.0 - 2.0 * s) * (2.0 * math.pi / nphi)  # Fejer's first rule
        return th, np.full(nt, nphi), np.zeros(nt), w, nphi
    ns = g[1]
    r = np.arange(1, 4 * ns)
    i = np.minimum(r, 4 * ns - r)
    cap = i < ns
    th = np.where(cap, 2.0 * np.arcsin(np.minimum(1.0, i / (math.sqrt(6.0) * ns))),
                  np.arccos(np.clip(4.0 / 3.0 - 2.0 * r / (3.0 * ns), -1.0, 1.0)))
    th = np.where(cap & (r > 2 * ns), math.pi - th, th)
    n = np.where(cap, 4 * i, 4 * ns)
    p0 = np.where(cap, math.pi / (4.0 * i), np.where((r - ns) % 2 == 0, math.pi / (4.0 * ns), 0.0))
    return th, n, p0, np.full(len(r), 4.0 * math.pi / (12.0 * ns * ns)), 4 * ns


def _bands(th, gmax):
    nrep = (len(th) + 1) // 2
    lo = np.searchsorted(th, th[:nrep] - gmax, "left")
    hi = np.searchsorted(th, th[:nrep] + gmax, "right") - 1
    return lo, hi


def _pairs(lo, hi, i0, i1):
    cnt = hi[i0:i1] - lo[i0:i1] + 1
    ii = np.repeat(np.arange(i0, i1), cnt)
    jj = np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt) + lo[ii]
    return ii, jj


def work(case):
    """Maps read and written once, profiles read once; real ring FFTs (2.5 n log2 n), the band sum
    (8 operations per ring pair, mode and map) and per kernel the cheaper of the cosine sum and the
    FFT of every ring pair's samples."""
    nbytes = flops = 0.0
    op = case["op"]
    for g in _grids(case):
        th, n, _, _, N = _rings(g)
        B = g[3]
        NH = N // 2 + 1
        npix = float(n.sum())
        nbytes += 4.0 * npix * B * (4 if op == "fit" else 2)
        fft = float(np.sum(2.5 * n * np.log2(n)))
        flops += fft * B * (4 if op == "fit" else 2)
        for k, gmax in _profiles(case):
            nbytes += 8.0 * len(k)
            lo, hi = _bands(th, gmax)
            ii, jj = _pairs(lo, hi, 0, len(lo))
            A = np.sin(0.5 * (th[ii] + th[jj])) ** 2
            D = np.sin(0.5 * (th[ii] - th[jj])) ** 2
            q = (math.sin(0.5 * gmax) ** 2 - D) / np.maximum(A - D, 1e-300)
            x = 2.0 * np.arcsin(np.sqrt(np.clip(q, 0.0, 1.0)))
            taps = np.floor(x * N / (2.0 * math.pi)) + 1.0
            gen = float(np.sum(np.minimum(2.0 * taps * NH, 2.5 * N * math.log2(N))))
            each = B if case["beams"] == 1 or op == "multi" else 1
            flops += (2 if op == "fit" else 1) * (gen + 8.0 * len(ii) * NH * each)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit result
def _analysis(x, n, p0, basic, N):
    """Ring spectra a_m, m = 0..N/2, of maps x [B, npix]: periodic beyond a ring's own modes, or with
    the BASIC window."""
    NH = N // 2 + 1
    m = torch.arange(NH, device=x.device)
    off = np.concatenate([[0], np.cumsum(n)])
    parts, order = [], []
    for ln in np.unique(n):
        rows = np.nonzero(n == ln)[0]
        ln = int(ln)
        split = np.split(rows, np.nonzero(np.diff(rows) > 1)[0] + 1)
        xr = torch.cat([x[:, off[s[0]]:off[s[-1] + 1]].reshape(x.shape[0], len(s), ln) for s in split], 1)
        a = torch.fft.fft(xr)[:, :, m % ln]
        ph = torch.tensor(p0[rows], device=x.device)[:, None] * m
        a = a * torch.polar(torch.ones_like(ph), -ph)
        if basic:
            a = a * torch.where(2 * m > ln, 0.0, torch.where((2 * m == ln) & (ln < N), 0.5, 1.0))
        parts.append(a)
        order.append(rows)
    inv = torch.tensor(np.argsort(np.concatenate(order)), device=x.device)
    return torch.cat(parts, 1)[:, inv]


def _synthesis(c, n, p0, basic, N):
    """Maps from the kernel-grid coefficients c [B, R, N/2 + 1] of every ring."""
    NH = N // 2 + 1
    off = np.concatenate([[0], np.cumsum(n)])
    parts, where = [], []
    for ln in np.unique(n):
        rows = np.nonzero(n == ln)[0]
        ln = int(ln)
        top = ln // 2 if basic else N // 2
        m = torch.arange(top + 1, device=c.device)
        ph = torch.tensor(p0[rows], device=c.device)[:, None] * m
        h = torch.where((m == 0) | (m == top), 0.5, 1.0).to(torch.float64)
        d = c[:, torch.tensor(rows, device=c.device), :top + 1] * torch.polar(h + 0 * ph, ph)
        z = torch.zeros(c.shape[0], len(rows), ln, dtype=d.dtype, device=c.device).index_add(2, m % ln, d)
        parts.append((2.0 * ln * torch.fft.ifft(z).real).reshape(c.shape[0], -1))
        where += [np.arange(off[r], off[r + 1]) for r in rows]
    inv = torch.empty(int(off[-1]), dtype=torch.int64, device=c.device)
    inv[torch.tensor(np.concatenate(where), device=c.device)] = torch.arange(int(off[-1]), device=c.device)
    return torch.cat(parts, 1)[:, inv]


class _Profile:
    """The tabulated profile: linear in u = 2 (1 - cos gamma) between knots, zero past the support."""

    def __init__(self, knots, gmax, dev):
        self.f = torch.tensor(knots, dtype=torch.float64, device=dev)
        t = torch.arange(len(knots), dtype=torch.float64, device=dev)
        self.u = 4.0 * torch.sin(0.5 * gmax * t / (len(knots) - 1)) ** 2
        self.gmax = gmax

    def hat(self, u):
        """(segment, position in it, inside the support) of squared chords u."""
        t = (torch.searchsorted(self.u, u, right=True) - 1).clamp(0, len(self.f) - 2)
        return t, (u - self.u[t]) / (self.u[t + 1] - self.u[t]), u <= self.u[-1]

    def __call__(self, u):
        t, lam, inside = self.hat(u)
        return torch.where(inside, self.f[t] + lam * (self.f[t + 1] - self.f[t]), 0.0)


def _blocks(lo, hi, N):
    i0 = 0
    while i0 < len(lo):
        i1 = i0 + 1
        while i1 < len(lo) and i1 - i0 < 64 and (hi[i0:i1 + 1] - lo[i0:i1 + 1] + 1).sum() * N < 3.0e7:
            i1 += 1
        yield i0, i1
        i0 = i1


def _chords(th, p0, n, ii, jj, N, dev):
    """Squared chords of the N kernel samples of ring pairs (i, j), taken at the pixel offset of
    equal-length rings, and that offset."""
    t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
    delta = t(np.where(n[ii] == n[jj], p0[ii] - p0[jj], 0.0))[:, None]
    x = 0.5 * (delta + 2.0 * math.pi / N * torch.arange(N, dtype=torch.float64, device=dev))
    s = torch.sin(x) ** 2
    A, D = t(np.sin(0.5 * (th[ii] + th[jj])) ** 2)[:, None], t(np.sin(0.5 * (th[ii] - th[jj])) ** 2)[:, None]
    return 4.0 * (D * torch.cos(x) ** 2 + A * s), delta


def _coefficients(K, delta, N):
    f = torch.fft.rfft(K) / N
    ph = delta * torch.arange(N // 2 + 1, device=K.device)
    return f.real * torch.cos(ph) + f.imag * torch.sin(ph)


def _band_sum(rho, ii, jj, i0, i1, u0, u1, A):
    """c [2 B, i1 - i0, NH] from coefficients rho of the pairs and spectra A [2 B, R, NH]: the maps
    and, with the rings in reverse order, their mirrors."""
    NH = rho.shape[1]
    at = torch.tensor((ii - i0) * (u1 - u0) + jj - u0, device=rho.device)
    dense = torch.zeros((i1 - i0) * (u1 - u0), NH, dtype=rho.dtype, device=rho.device).index_copy(0, at, rho)
    a = torch.view_as_real(A[:, u0:u1].contiguous()).permute(2, 1, 0, 3).reshape(NH, u1 - u0, -1)
    c = torch.bmm(dense.view(i1 - i0, u1 - u0, NH).permute(2, 0, 1), a)
    return torch.view_as_complex(c.view(NH, i1 - i0, -1, 2).permute(2, 1, 0, 3).contiguous())


def _pole_chords(th, n, p0, gmax, dev):
    """Per pole ring: its pixels' squared chords to the pixels of the rings inside the support, and
    where those pixels start in the map."""
    off = np.concatenate([[0], np.cumsum(n)])
    for i, rows in ((0, np.nonzero(th <= th[0] + gmax)[0]), (len(th) - 1, np.nonzero(th >= th[-1] - gmax)[0])):
        tq = np.repeat(th[rows], n[rows])
        pq = np.concatenate([p0[r] + 2.0 * math.pi * np.arange(n[r]) / n[r] for r in rows])
        tq, pq = torch.tensor(tq, device=dev), torch.tensor(pq, device=dev)
        pp = torch.tensor(p0[i] + 2.0 * math.pi * np.arange(n[i]) / n[i], device=dev)[:, None]
        x = 0.5 * (pp - pq)
        u = 4.0 * (torch.sin(0.5 * (th[i] - tq)) ** 2 * torch.cos(x) ** 2 + torch.sin(0.5 * (th[i] + tq)) ** 2 * torch.sin(x) ** 2)
        yield slice(int(off[i]), int(off[i + 1])), slice(int(off[rows[0]]), int(off[rows[-1] + 1])), u


def _exact_maps(g, prof, x, basic, weights=None, grad=None):
    """The convolution of maps x [B, npix] (float64): one profile, one per map, or with weights the
    weighted sum over the profiles.  With grad also the gradients of x and of the knots."""
    th, n, p0, w, N = _rings(g)
    dev, B, R = x.device, x.shape[0], len(th)
    wt = torch.tensor(w, device=dev)[None, :, None]
    fit = grad is not None
    x = x.requires_grad_(fit)
    A = _analysis(x, n, p0, basic, N) * wt
    a = A.detach()
    a2 = torch.cat([a, a.flip(1)])  # the mirrors' band sums share the coefficients
    c = torch.zeros(B, R, N // 2 + 1, dtype=torch.complex128, device=dev)
    per_map = weights is None and len(prof) > 1
    P = [_Profile(k, gm, dev) for k, gm in prof]
    bands = [_bands(th, p.gmax) for p in P]

    def maps_of(k):
        return slice(k, k + 1) if per_map else slice(0, B)

    for k, p in enumerate(P):
        s, sc = maps_of(k), 1.0 if weights is None else float(weights[k])
        nb = s.stop - s.start
        ak = torch.cat([a2[:B][s], a2[B:][s]])
        for i0, i1 in _blocks(*bands[k], N):
            ii, jj = _pairs(*bands[k], i0, i1)
            u, delta = _chords(th, p0, n, ii, jj, N, dev)
            cb = sc * _band_sum(_coefficients(p(u), delta, N), ii, jj, i0, i1, jj.min(), jj.max() + 1, ak)
            c[s, i0:i1] += cb[:nb]
            south = np.array([i for i in range(i0, i1) if R - 1 - i != i])
            if len(south):
                c[s, torch.tensor(R - 1 - south, device=dev)] += cb[nb:, torch.tensor(south - i0, device=dev)]
    c = c.requires_grad_(fit)
    y = _synthesis(c, n, p0, basic, N)
    out = y.detach().clone()
    poles = g[0] == "healpix"
    for k, p in enumerate(P if poles else []):
        s, sc = maps_of(k), 1.0 if weights is None else float(weights[k])
        for po, pi, u in _pole_chords(th, n, p0, p.gmax, dev):
            v = sc * w[0] * x.detach()[s, pi] @ p(u).T
            out[s, po] = v if k == 0 or per_map else out[s, po] + v
    if not fit:
        return out
    gr = grad.clone()
    if poles:  # the hybrid values of the pole rings are replaced
        gr[:, :n[0]] = 0.0
        gr[:, -n[-1]:] = 0.0
    y.backward(gr)
    del y
    gc = c.grad
    gc2 = torch.cat([gc, gc.flip(1)])
    gA = torch.zeros_like(a)
    gk = torch.zeros(len(P), len(prof[0][0]), dtype=torch.float64, device=dev)

    def deposit(k, p, u, gK):
        t, lam, inside = p.hat(u)
        at = inside & (gK != 0)
        t, lam, v = t[at], lam[at], gK[at]
        T = gk.shape[1]
        gk[k] += torch.bincount(t, (1.0 - lam) * v, T) + torch.bincount(t + 1, lam * v, T)

    for k, p in enumerate(P):
        s = maps_of(k)
        nb = s.stop - s.start
        for i0, i1 in _blocks(*bands[k], N):
            ii, jj = _pairs(*bands[k], i0, i1)
            u, delta = _chords(th, p0, n, ii, jj, N, dev)
            K = p(u).requires_grad_(True)
            u0, u1 = int(jj.min()), int(jj.max()) + 1
            ak = torch.cat([a2[:B][s, u0:u1], a2[B:][s, u0:u1]]).requires_grad_(True)
            cb = _band_sum(_coefficients(K, delta, N), ii - 0, jj - u0, i0, i1, 0, u1 - u0, ak)
            gb = torch.cat([gc2[:B][s, i0:i1], gc2[B:][s, i0:i1]]).clone()
            mid = [i - i0 for i in range(i0, i1) if R - 1 - i == i]
            gb[nb:, mid] = 0.0  # the middle ring is its own mirror
            cb.backward(gb)
            gA[s, u0:u1] += ak.grad[:nb]
            gA[s, R - u1:R - u0] += ak.grad[nb:].flip(1)
            deposit(k, p, u, K.grad)
    A.backward(gA)
    gx = x.grad.clone()
    for k, p in enumerate(P if poles else []):
        s = maps_of(k)
        for po, pi, u in _pole_chords(th, n, p0, p.gmax, dev):
            gx[s, pi] += w[0] * grad[s, po] @ p(u)
            deposit(k, p, u, w[0] * grad[s, po].T @ x.detach()[s, pi])
    return out, gx, gk


def exact(case, seed):
    if not torch.cuda.is_available() and work(case)["flops"] > 2.0e9:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    maps, grad = _maps(case, seed, dev)
    prof = _profiles(case)
    weights = _weights(case, seed) if case["op"] == "multi" else None
    out = []
    for g, x in zip(_grids(case), maps):
        r = _exact_maps(g, prof, x.double(), case["basic"], weights, grad[0].double() if grad else None)
        if case["op"] == "fit":
            return r
        out.append(r)
    return out if case["op"] == "batch" else out[0]
