"""Performance cases: the work that a user of the library has it do, through its public entry points.

A case is a dict of plain values.  `kind` names the call:

  zeta            Context.zeta_ell, the whole measurement of one catalogue
  batch           Context.batch, many small catalogues of uneven size in one launch
  catalogue       Context.assign, fft_r2c and sort_particles: the steps taken once per catalogue
  fields          Context.reconstruct_alm, the fields of one (l, m)
  grid_sum        Context.sum_grid, the node or the Gamma form of one (l, m)
  particle_sum    Context.sum_particles, the particle form of one (l, m)
  xi              Context.xi, the 2PCF in both forms
  grad_node       Context.backward_node, the gradient in the density contrast
  grad_particles  Context.backward_particles, the gradient in the particle positions

Grids, particle counts, bins and multipoles come from the named workloads (workloads.py), the tests
and the benchmark.  Inputs are log-normal mocks like those of mocks.py (unit-variance Gaussian field,
P(k) ~ k^-1.5), drawn on the GPU so that they are quick to make.  exact() restates the method in
float64 with torch alone.
"""
import math

import numpy as np
import torch

from paper_2507_15209_gb300.zeta import Context

FORMS = ("node", "gamma", "particle")


def listed():
    return [
        # the smallest whole measurement: 20k galaxies, every summation form; a few hundred short launches
        dict(name="zeta_n64_all_forms", kind="zeta", n=64, box=500.0, np=20_000, dsup=2, lmax=4, nb=8, r_lo=10.0,
             r_hi=90.0, forms="node,gamma,particle", weights=False),
        # an ordinary survey mock, the particle form at the paper's resolution (256^3, l <= 10)
        dict(name="zeta_n256_particle", kind="zeta", n=256, box=1000.0, np=2_000_000, dsup=4, lmax=10, nb=15,
             r_lo=5.0, r_hi=150.0, forms="particle", weights=False),
        # a covariance run: many small mocks of uneven size in one call
        dict(name="batch_n64", kind="batch", n=64, box=500.0, np=300_001, ncat=8, dsup=2, lmax=4, nb=8, r_lo=10.0,
             r_hi=90.0, forms="node,particle", weights=False),
        # a catalogue read in: density grid, its transform and the tiling, with galaxy weights and a ragged count
        dict(name="catalogue_n256", kind="catalogue", n=256, box=1000.0, np=2_000_003, dsup=4, lmax=0, nb=1,
             r_lo=5.0, r_hi=150.0, weights=True),
        # the fields of one (l, m) on the largest grid, the step that repeats (lmax + 1)^2 times
        dict(name="fields_n512_b20", kind="fields", n=512, box=2000.0, np=16_000_000, dsup=4, lmax=7, nb=20, r_lo=5.0,
             r_hi=200.0, l=7, m=-5, weights=False),
        # the same on an ordinary grid with an odd number of bins
        dict(name="fields_n128_b13", kind="fields", n=128, box=500.0, np=250_000, dsup=4, lmax=4, nb=13, r_lo=5.0,
             r_hi=75.0, l=4, m=3, weights=False),
        # the grid sum in the node form on the largest grid
        dict(name="node_n512_b20", kind="grid_sum", form="node", gram="fp32", n=512, box=2000.0, np=16_000_000, dsup=4,
             lmax=2, nb=20, r_lo=5.0, r_hi=200.0, l=2, m=1, weights=False),
        # the grid sum in the connection-coefficient form, cubic B-spline
        dict(name="gamma_n128_b15", kind="grid_sum", form="gamma", gram="fp32", n=128, box=500.0, np=250_000, dsup=4,
             lmax=2, nb=15, r_lo=5.0, r_hi=75.0, l=2, m=0, weights=False),
        # the particle sum on the largest grid and catalogue
        dict(name="particles_n512_np16m", kind="particle_sum", n=512, box=2000.0, np=16_000_000, dsup=4, lmax=2, nb=20,
             r_lo=5.0, r_hi=200.0, l=2, m=-1, weights=False),
        # the 2PCF of a survey mock beside its 3PCF
        dict(name="xi_n256", kind="xi", n=256, box=1000.0, np=2_000_000, dsup=4, lmax=0, nb=15, r_lo=5.0, r_hi=150.0,
             weights=False),
        # field-level inference: the gradient in the density grid
        dict(name="grad_node_n256", kind="grad_node", n=256, box=1000.0, np=1_000_000, dsup=4, lmax=6, nb=10, r_lo=10.0,
             r_hi=110.0, weights=False),
        # field-level inference: the gradient in the particle positions
        dict(name="grad_particles_n256", kind="grad_particles", n=256, box=1000.0, np=1_000_000, dsup=4, lmax=6, nb=10,
             r_lo=10.0, r_hi=110.0, weights=False),
    ]


def draw(rng):
    kind = rng.choice(["zeta", "zeta", "batch", "catalogue", "fields", "fields", "grid_sum", "grid_sum",
                       "particle_sum", "xi", "grad_node", "grad_particles"])
    n = rng.choice({"batch": [16, 32, 64], "zeta": [32, 64, 128, 256], "grad_node": [32, 64, 128, 256],
                    "grad_particles": [32, 64, 128, 256], "xi": [64, 128, 256, 512]}.get(kind, [64, 128, 256, 512]))
    small = n <= 128
    box = rng.choice([500.0, 1000.0, 1500.0]) if small else rng.choice([1000.0, 2000.0])
    # galaxy catalogues: about 0.01 to 0.12 particles per cell on large grids, a few on the smallest
    dens = math.exp(rng.uniform(math.log(0.01), math.log(0.12 if n >= 128 else 0.5)))
    npart = max(997, int(dens * n ** 3) | 1)
    dsup = rng.choice([2, 4, 4, 3])
    nb = rng.randint(1, 20)
    lmax = rng.randint(0, 10)
    case = dict(kind=kind, n=n, box=box, np=npart, dsup=dsup, r_lo=0.01 * box, r_hi=rng.uniform(0.1, 0.18) * box,
                weights=rng.random() < 0.3)
    if kind == "zeta":
        forms = rng.choice(["particle", "node", "node,particle"])
        if n <= 64 and rng.random() < 0.3:
            forms = "node,gamma,particle"
        if n == 256:
            lmax = rng.randint(0, 6)
            nb = min(nb, 15)
        case.update(forms=forms)
    elif kind == "batch":
        lmax = rng.randint(0, 4)
        nb = rng.randint(1, 10)
        case.update(ncat=rng.randint(2, 9), forms=rng.choice(["particle", "node,particle"]))
        case["np"] = max(case["ncat"] * 997, int(rng.uniform(0.02, 0.3) * n ** 3) * case["ncat"] | 1)
    elif kind in ("catalogue", "xi"):
        lmax = 0
    elif kind in ("fields", "grid_sum", "particle_sum"):
        lmax = rng.randint(0, 7)
        case.update(l=lmax, m=rng.randint(-lmax, lmax))
        if kind != "fields" or n < 512:
            nb = rng.randint(1, 32 if n < 512 else 20)
        if kind == "grid_sum":
            case.update(form=rng.choice(["node", "node", "gamma"]), gram="fp32")
            if case["form"] == "gamma":
                case["n"] = n = rng.choice([32, 64, 128])
                case.update(np=max(997, int(dens * n ** 3) | 1))
                nb = min(nb, 15)
            else:
                case["gram"] = rng.choice(["fp32", "fp32", "fp32", "bf16x3"])
    else:
        case["dsup"] = rng.choice([2, 4])
        nb = rng.randint(1, 10)
        lmax = rng.randint(0, 4 if n == 256 else 6)
    case.update(lmax=lmax, nb=nb)
    return case


# ---- inputs ------------------------------------------------------------------------------------
def _edges(case):
    return np.linspace(case["r_lo"], case["r_hi"], case["nb"] + 1)


def _catalogue(case, seed, npart=None):
    """A log-normal mock on the GPU: float32 (np, 4).  The cells are drawn from an integer
    cumulative density, so the same seed gives the same particles."""
    n, box, npart = case["n"], case["box"], npart or case["np"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    wk = torch.fft.rfftn(torch.randn((n, n, n), device="cuda", generator=g))
    i = torch.fft.fftfreq(n, 1.0 / n, device="cuda")
    k2 = i[:, None, None] ** 2 + i[None, :, None] ** 2 + i[None, None, : n // 2 + 1].abs() ** 2
    k2[0, 0, 0] = 1.0
    wk *= k2 ** (-1.5 / 4)
    wk[0, 0, 0] = 0.0
    rho = torch.fft.irfftn(wk, s=(n, n, n))
    rho = torch.exp(rho / rho.std() - 0.5)
    cdf = torch.cumsum((rho.reshape(-1) * 65536.0).long(), 0)
    del wk, k2, rho
    u = (torch.rand(npart, device="cuda", generator=g, dtype=torch.float64) * float(cdf[-1])).long()
    cell = torch.searchsorted(cdf, u, right=True).clamp_(max=n ** 3 - 1)
    del cdf, u
    ijk = torch.stack([cell % n, (cell // n) % n, cell // (n * n)], 1)
    pos = ((ijk + torch.rand((npart, 3), device="cuda", generator=g, dtype=torch.float64)) * (box / n)).float()
    pos[pos >= box] = 0.0
    out = torch.ones((npart, 4), device="cuda")
    out[:, :3] = pos
    if case["weights"]:
        out[:, 3] = torch.rand(npart, device="cuda", generator=g) + 0.5
    return out


def _sizes(case, seed):
    """Uneven catalogue sizes of a batch, summing to case["np"]."""
    f = np.random.Generator(np.random.PCG64(int(seed))).uniform(0.3, 1.7, case["ncat"])
    cuts = np.round(np.cumsum(f / f.sum()) * case["np"]).astype(np.int64)
    return np.diff(np.concatenate([[0], cuts]))


def _daub_table():
    """The genus-4 Daubechies function at k / 2^10, from its two-scale relation."""
    s = math.sqrt(3.0)
    c = np.array([1 + s, 3 + s, 3 - s, 1 - s]) / 4.0
    v = np.array([0.0, (1 + s) / 2, (1 - s) / 2, 0.0])
    for j in range(10):
        m, step = 3 << (j + 1), 1 << j
        new = np.zeros(m + 1)
        new[::2] = v
        odd = np.arange(1, m, 2)
        for i in range(4):
            src = odd - i * step
            ok = (src >= 0) & (src <= 3 * step)
            new[odd[ok]] += c[i] * v[src[ok]]
        v = new
    return v


def _stencil(x, n, box, dsup, grad=False):
    """Per axis: first node and the weights (dsup rows) of the particles at x (float64)."""
    u = x * (n / box)
    c = torch.floor(u)
    t = u - c
    if dsup == 3:
        tab = torch.from_numpy(_daub_table()).to(x.device)
        i = (t * 1024).long().clamp(0, 1023)
        f = t * 1024 - i
        w = [torch.lerp(tab[i + (2 - o) * 1024], tab[i + 1 + (2 - o) * 1024], f) for o in range(3)]
        return c.long() - 2, w
    if dsup == 2:
        w, d = [1 - t, t], [-torch.ones_like(t), torch.ones_like(t)]
    else:
        w = [(1 - t) ** 3 / 6, (3 * t ** 3 - 6 * t * t + 4) / 6, (-3 * t ** 3 + 3 * t * t + 3 * t + 1) / 6, t ** 3 / 6]
        d = [-0.5 * (1 - t) ** 2, 1.5 * t * t - 2 * t, -1.5 * t * t + t + 0.5, 0.5 * t * t]
    return (c.long() - (dsup // 2 - 1), w, [v * (n / box) for v in d]) if grad else (c.long() - (dsup // 2 - 1), w)


def _nodes(case, pos, grad=False):
    """(flat node index, weight[, its gradient (np, 3)]) of every stencil node of the particles."""
    n = case["n"]
    ax = [_stencil(pos[:, d].double(), n, case["box"], case["dsup"], grad) for d in range(3)]
    for oz in range(case["dsup"]):
        for oy in range(case["dsup"]):
            for ox in range(case["dsup"]):
                o = (ox, oy, oz)
                i, j, k = ((ax[d][0] + o[d]) % n for d in range(3))
                w = [ax[d][1][o[d]] for d in range(3)]
                at = (k * n + j) * n + i
                if not grad:
                    yield at, w[0] * w[1] * w[2]
                else:
                    g = [ax[d][2][o[d]] for d in range(3)]
                    yield at, w[0] * w[1] * w[2], torch.stack([g[0] * w[1] * w[2], w[0] * g[1] * w[2],
                                                               w[0] * w[1] * g[2]], 1)


def _contrast(case, parts):
    """delta in float64: the basis assignment of the catalogue over its mean, less one (summed as
    integers, so the order of the particles does not matter)."""
    n = case["n"]
    eps = torch.zeros(n ** 3, dtype=torch.int64, device="cuda")
    for p in parts.split(4_000_000):
        for at, w in _nodes(case, p):
            eps.index_add_(0, at, torch.round(w * p[:, 3].double() * 2.0 ** 40).long())
    return (eps.double() * (n ** 3 / 2.0 ** 40 / parts[:, 3].double().sum()) - 1.0).reshape(n, n, n)


# ---- the method in plain torch -------------------------------------------------------------------
def _jn(l, x):
    """Spherical Bessel j_l(x), x >= 0: upward where x > l, Miller's downward recurrence below."""
    big = x > l + 1
    xu = torch.where(big, x, torch.full_like(x, l + 2.0))
    a, b = torch.sin(xu) / xu, torch.sin(xu) / xu ** 2 - torch.cos(xu) / xu
    up = a
    for k in range(l):
        up = b
        a, b = b, (2 * k + 3) / xu * b - a
    xd = torch.where(big, torch.full_like(x, 1.0), x).clamp(min=1e-2)
    hi, lo, got = torch.zeros_like(x), torch.full_like(x, 1e-250), None
    j1 = None
    for k in range(l + 40, -1, -1):  # lo = j_k up to scale
        if k == l:
            got = lo
        if k == 1:
            j1 = lo
        if k == 0:
            break
        hi, lo = lo, (2 * k + 1) / xd * lo - hi
    s, c = torch.sin(xd), torch.cos(xd)
    t0, t1 = s / xd, s / xd ** 2 - c / xd
    scale = torch.where(t0.abs() > t1.abs(), t0 / lo, t1 / j1)
    return torch.where(big, up, got * scale)


def _radial(case, l):
    """The r^2-weighted shell average of j_l(k r) of every bin, by integer |n|^2: (n2, nb) float64."""
    n, box, e = case["n"], case["box"], _edges(case)
    k = 2 * math.pi / box * torch.sqrt(torch.arange(3 * (n // 2 - 1) ** 2 + 1, device="cuda", dtype=torch.float64))
    xg, wg = np.polynomial.legendre.leggauss(24)
    out = torch.zeros((len(k), case["nb"]), dtype=torch.float64, device="cuda")
    for b in range(case["nb"]):
        cuts = np.linspace(e[b], e[b + 1], max(1, math.ceil(float(k[-1]) * (e[b + 1] - e[b]) / 8.0)) + 1)
        for lo, hi in zip(cuts[:-1], cuts[1:]):
            for x, w in zip(xg, wg):
                r = 0.5 * (lo + hi) + 0.5 * (hi - lo) * x
                out[:, b] += (0.5 * (hi - lo) * w * r * r) * _jn(l, k * r)
        out[:, b] *= 3.0 / (e[b + 1] ** 3 - e[b] ** 3)
    out[0] = 1.0 if l == 0 else 0.0
    return out


def _freq(n):
    i = torch.arange(n, device="cuda")
    f = torch.where(i < n // 2, i, i - n)
    nx, ny, nz = f[None, None, : n // 2], f[None, :, None], f[:, None, None]
    keep = (ny != -(n // 2)) & (nz != -(n // 2))
    return nx, ny, nz, keep, torch.where(keep, nx * nx + ny * ny + nz * nz, 0)


def _ylm(case, l, m):
    """sqrt(4 pi) R_lm of the half spectrum's directions in float64, zero on the Nyquist planes."""
    nx, ny, nz, keep, n2 = _freq(case["n"])
    r = torch.sqrt(n2.double()).clamp(min=0.5)
    ct, sx, sy = nz / r, nx / r, ny / r
    a = abs(m)
    cr, ci = torch.ones_like(r), torch.zeros_like(r)
    for _ in range(a):
        cr, ci = cr * sx - ci * sy, cr * sy + ci * sx
    q = math.sqrt(2.0 if a else 1.0)
    for k in range(1, a + 1):
        q *= math.sqrt((2 * k - 1.0) / (2 * k))
    p0, p1 = torch.zeros_like(r), torch.full_like(r, q)  # associated Legendre, Schmidt's normalisation
    for k in range(a + 1, l + 1):
        p0, p1 = p1, ((2 * k - 1) * ct * p1 - math.sqrt((k - 1.0) ** 2 - a * a) * p0) / math.sqrt(k * k - a * a)
    out = math.sqrt(2 * l + 1) * p1 * (ci if m < 0 else cr)
    return torch.where(keep & ((n2 > 0) | (l == 0)), out, torch.zeros_like(out))


def _window(case, l, m, radial, b, ylm, n2):
    return ylm * radial[:, b][n2]


def _fields(case, dhat, l, m, radial, dtype=torch.complex128):
    """a_lm of every bin: a list of (n, n, n) real grids, from the half spectrum dhat (n, n, n/2)."""
    n = case["n"]
    ylm, n2 = _ylm(case, l, m), _freq(n)[4]
    full = torch.zeros((n, n, n // 2 + 1), dtype=dtype, device="cuda")
    for b in range(case["nb"]):
        full[..., : n // 2] = dhat * (_window(case, l, m, radial, b, ylm, n2) * (1j ** l)).to(dtype)
        yield torch.fft.irfftn(full, s=(n, n, n))


def _interleave(case, fields, dtype):
    n, nb = case["n"], case["nb"]
    out = torch.zeros(((nb + 3) // 4, n, n, n, 4), dtype=dtype, device="cuda")
    for b, a in enumerate(fields):
        out[b // 4, ..., b % 4] = a
    return out


def _points(case, fields, parts, grad=False):
    """f_b at the particles (np, nb), with grad also its gradient (np, nb, 3)."""
    n, nb = case["n"], case["nb"]
    flat = torch.empty((n ** 3, nb), dtype=torch.float64, device="cuda")
    for b, a in enumerate(fields):
        flat[:, b] = a.reshape(-1)
    vals, grads = [], []
    for p in parts.split(1_000_000):
        f = torch.zeros((len(p), nb), dtype=torch.float64, device="cuda")
        g = torch.zeros((len(p), nb, 3), dtype=torch.float64, device="cuda") if grad else None
        for node in _nodes(case, p, grad):
            v = flat[node[0]]
            f += node[1][:, None] * v
            if grad:
                g += v[:, :, None] * node[2][:, None, :]
        vals.append(f)
        grads.append(g)
    return (torch.cat(vals), torch.cat(grads)) if grad else torch.cat(vals)


def _half(delta):
    return torch.fft.rfftn(delta)[..., : delta.shape[0] // 2]


def _mass_hat(case):
    """The DFT of the basis's mass matrix per axis."""
    n, m = case["n"], {2: [2 / 3, 1 / 6], 3: [1.0], 4: [151 / 315, 397 / 1680, 1 / 42, 1 / 5040]}[case["dsup"]]
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    return torch.full_like(k, m[0]) + sum(2 * v * torch.cos(2 * math.pi * a * k / n) for a, v in enumerate(m) if a)


def _uniform(case, dhat):
    """Mode weights of the uniform term summed per |n|^2."""
    n = case["n"]
    _, _, _, keep, n2 = _freq(n)
    h = _mass_hat(case)
    w = dhat.abs() ** 2 * (h[:, None, None] * h[None, :, None] * h[None, None, : n // 2]) * keep
    w[..., 1:] *= 2
    return torch.zeros(3 * (n // 2 - 1) ** 2 + 1, dtype=torch.float64, device="cuda").index_add_(0, n2.reshape(-1), w.reshape(-1))


def _gamma_points(dsup):
    """Per axis (weights, filters): the point k of a cell (or the eigen-index k of a node) has the
    value sum_o filters[k][o] a(l + first + o); first; whether the primary vertex is filtered too."""
    if dsup != 3:
        q = 2 if dsup == 2 else 5
        x, w = np.polynomial.legendre.leggauss(q)
        _, b = _stencil(torch.from_numpy((x + 1) / 2), 1, 1.0, dsup)
        return w / 2, np.stack([v.numpy() for v in b], 1), -(dsup // 2 - 1), True
    s = math.sqrt(3.0)
    h = np.array([1 + s, 3 + s, 3 - s, 1 - s]) / (4 * math.sqrt(2.0))
    at = {(a, b): i for i, (a, b) in enumerate((a, b) for a in range(-2, 3) for b in range(-2, 3) if abs(a - b) < 3)}
    rows = np.zeros((len(at) + 5, len(at)))
    rhs = np.zeros(len(at) + 5)
    rhs[len(at) + 2] = 1.0  # sum_b Gamma(0, b) = 1, the other rows sum to 0 (an orthonormal basis)
    for (a, b), i in at.items():
        rows[i, i] -= 1.0
        rows[len(at) + a + 2, i] = 1.0
        for u in range(4):
            for v in range(4):
                for w in range(4):
                    j = at.get((2 * a + v - u, 2 * b + w - u))
                    if j is not None:
                        rows[i, j] += math.sqrt(2.0) * h[u] * h[v] * h[w]
    x = np.linalg.lstsq(rows, rhs, rcond=None)[0]
    gm = np.zeros((5, 5))
    for (a, b), i in at.items():
        gm[a + 2, b + 2] = x[i]
    lam, vec = np.linalg.eigh(0.5 * (gm + gm.T))
    return lam, vec.T, -2, False


def _gamma_sum(case, delta, fields):
    """The connection-coefficient form of one (l, m), as its separable points."""
    w, f, first, filt = _gamma_points(case["dsup"])
    nb = case["nb"]
    a = torch.stack(list(fields) + [delta])

    def along(x, k, axis):
        return sum(float(f[k][o]) * torch.roll(x, -(first + o), axis) for o in range(f.shape[1]))

    out = torch.zeros((nb, nb), dtype=torch.float64, device="cuda")
    for kz in range(len(w)):
        az = along(a, kz, 1)
        for ky in range(len(w)):
            ay = along(az, ky, 2)
            for kx in range(len(w)):
                v = along(ay, kx, 3)
                d = (v[nb] if filt else delta).reshape(1, -1) * float(w[kx] * w[ky] * w[kz])
                v = v[:nb].reshape(nb, -1)
                out += (v * d) @ v.T
    return out / delta.numel()


def _zeta(case, parts, delta=None):
    """{form: (lmax + 1, nb, nb)} of a catalogue."""
    forms = case["forms"].split(",")
    delta = _contrast(case, parts) if delta is None else delta
    dhat = _half(delta)
    out = {f: torch.zeros((case["lmax"] + 1, case["nb"], case["nb"]), dtype=torch.float64, device="cuda") for f in forms}
    wsum = parts[:, 3].double().sum()
    hist = _uniform(case, dhat)
    for l in range(case["lmax"] + 1):
        rad = _radial(case, l)
        if "particle" in forms:
            out["particle"][l] -= (2 * l + 1) / float(case["n"]) ** 6 * (rad * hist[:, None]).T @ rad
        for m in range(-l, l + 1):
            a = list(_fields(case, dhat, l, m, rad))
            if "node" in forms:
                v = torch.stack(a).reshape(case["nb"], -1)
                out["node"][l] += (v * delta.reshape(1, -1)) @ v.T / delta.numel()
            if "gamma" in forms:
                out["gamma"][l] += _gamma_sum(case, delta, a)
            if "particle" in forms:
                f = _points(case, a, parts)
                out["particle"][l] += (f * parts[:, 3:].double()).T @ f / wsum
    return out


def _grad_node(case, delta, weights):
    n = case["n"]
    dhat = _half(delta)
    q = torch.zeros_like(delta)
    gk = torch.zeros((n, n, n // 2 + 1), dtype=torch.complex128, device="cuda")
    for l in range(case["lmax"] + 1):
        s = 0.5 * (weights[l] + weights[l].T)
        rad = _radial(case, l)
        for m in range(-l, l + 1):
            a = torch.stack(list(_fields(case, dhat, l, m, rad)))
            sa = torch.einsum("ij,jxyz->ixyz", s, a)
            q += (sa * a).sum(0)
            gk[..., : n // 2] += _transpose(case, l, m, rad, (2 * delta * h for h in sa))
    return (q + torch.fft.irfftn(gk, s=(n, n, n))) / delta.numel()


def _transpose(case, l, m, rad, h):
    """(-1)^l sum_b K_b DFT(h_b) on the half spectrum."""
    ylm, n2 = _ylm(case, l, m), _freq(case["n"])[4]
    return sum(_half(x) * (_window(case, l, m, rad, b, ylm, n2) * ((-1j) ** l)) for b, x in enumerate(h))


def _grad_particles(case, parts, weights):
    n = case["n"]
    w = parts[:, 3].double()
    wsum = w.sum()
    dhat = _half(_contrast(case, parts))
    mh = _mass_hat(case)
    mh = mh[:, None, None] * mh[None, :, None] * mh[None, None, : n // 2]
    n2 = _freq(n)[4]
    direct = torch.zeros((len(parts), 3), dtype=torch.float64, device="cuda")
    gk = torch.zeros((n, n, n // 2 + 1), dtype=torch.complex128, device="cuda")
    for l in range(case["lmax"] + 1):
        s = 0.5 * (weights[l] + weights[l].T)
        rad = _radial(case, l)
        # the uniform term's share: (-1)^l i^(2l) = 1, and the R_lm R_lm sum to (2 l + 1) / (4 pi)
        gk[..., : n // 2] -= 2.0 / n ** 3 * (2 * l + 1) * dhat * mh * (torch.einsum("ib,bc,ic->i", rad, s, rad))[n2] * _freq(n)[3]
        for m in range(-l, l + 1):
            f, df = _points(case, list(_fields(case, dhat, l, m, rad)), parts, grad=True)
            c = (2 * w / wsum)[:, None] * (f @ s)
            direct += torch.einsum("pb,pbd->pd", c, df)
            del f, df
            h = torch.zeros((n ** 3, case["nb"]), dtype=torch.float64, device="cuda")
            for at, wt in _nodes(case, parts):
                h.index_add_(0, at, wt[:, None] * c)
            gk[..., : n // 2] += _transpose(case, l, m, rad, (h[:, b].reshape(n, n, n) for b in range(case["nb"])))
    g = torch.fft.irfftn(gk, s=(n, n, n)).reshape(-1)
    via = torch.zeros_like(direct)
    for at, _, dw in _nodes(case, parts, grad=True):
        via += g[at][:, None] * dw
    return direct + (n ** 3 / wsum) * w[:, None] * via


# ---- the cases -----------------------------------------------------------------------------------
def _inputs(case, seed):
    """Everything a user's program has in hand before the call, on the GPU."""
    kind = case["kind"]
    if kind == "batch":
        sizes = _sizes(case, seed)
        return dict(parts=torch.cat([_catalogue(case, 1000 * seed + i, int(s)) for i, s in enumerate(sizes)]), sizes=sizes)
    parts = _catalogue(case, seed)
    if kind in ("zeta", "catalogue", "xi"):
        return dict(parts=parts)
    out = {}
    if kind in ("grad_node", "grad_particles"):
        g = np.random.Generator(np.random.PCG64(int(seed)))
        out["weights"] = g.standard_normal((case["lmax"] + 1, case["nb"], case["nb"]))
    if kind in ("particle_sum", "grad_particles"):
        out["parts"] = parts
    if kind == "grad_particles":
        return out
    delta = _contrast(case, parts).float()
    if kind in ("grid_sum", "grad_node"):
        out["delta"] = delta
    if kind in ("fields", "grid_sum", "particle_sum"):
        dhat = _half(delta).contiguous()
        if kind == "fields":
            out["dhat"] = torch.view_as_real(dhat)
        else:
            rad = _radial(case, case["l"])
            out["alm"] = _interleave(case, _fields(case, dhat, case["l"], case["m"], rad, torch.complex64), torch.float32)
    return out


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case)
    kind, nb = case["kind"], case["nb"]
    forms = {"zeta": case.get("forms", "").split(","), "batch": case.get("forms", "").split(","), "xi": ["node", "particle"],
             "particle_sum": ["particle"], "catalogue": ["particle"], "grad_node": ["node", "backward"],
             "grad_particles": ["particle", "backward"]}.get(kind, ["node", "gamma"])
    npart = int(s["sizes"].max()) if kind == "batch" else len(s["parts"]) if "parts" in s else 0
    ctx = Context(case["n"], case["box"], case["dsup"], case["lmax"], _edges(case), gram=case.get("gram", "fp32"),
                  np_max=npart, forms=forms, ws_copies=4 if kind == "batch" else 1)
    s.update(ctx=ctx, forms=tuple(forms))
    if kind == "batch":
        s["offsets"] = np.concatenate([[0], np.cumsum(s["sizes"])])
        s["out"] = torch.empty((case["ncat"], len(forms), case["lmax"] + 1, nb, nb), dtype=torch.float64, device="cuda")
    if kind == "fields":
        s["out"] = torch.empty(((nb + 3) // 4, case["n"], case["n"], case["n"], 4), device="cuda")
    if kind == "particle_sum":
        s["sorted"], s["start"] = ctx.sort_particles(s["parts"])
        s["wsum"] = s["parts"][:, 3].double().sum().reshape(1)
    return s


def run(state):
    s, ctx = state, state["ctx"]
    kind = s["case"]["kind"]
    if kind == "zeta":
        return ctx.zeta_ell(particles=s["parts"], forms=s["forms"])
    if kind == "batch":
        return ctx.batch(s["parts"], s["offsets"], forms=s["forms"], out=s["out"])
    if kind == "catalogue":
        delta, wsum = ctx.assign(s["parts"])
        dhat = ctx.fft_r2c(delta)
        srt, start = ctx.sort_particles(s["parts"])
        return {"delta": delta, "dhat": dhat, "sorted": srt, "start": start, "wsum": wsum}
    if kind == "fields":
        return ctx.reconstruct_alm(s["dhat"], s["case"]["l"], s["case"]["m"], out=s["out"])
    if kind == "grid_sum":
        return ctx.sum_grid(s["delta"], s["alm"], form=s["case"]["form"])
    if kind == "particle_sum":
        return ctx.sum_particles(s["sorted"], s["start"], s["wsum"], s["alm"])
    if kind == "xi":
        return ctx.xi(particles=s["parts"], forms=("node", "particle"))
    if kind == "grad_node":
        return ctx.backward_node(s["delta"], s["weights"])
    return ctx.backward_particles(s["parts"], s["weights"])


def work(case):
    n, nb, npart, kind = case["n"], case["nb"], case["np"], case["kind"]
    ng, sten = n ** 3, case["dsup"] ** 3
    lm, lanes = (case["lmax"] + 1) ** 2, 4 * ((nb + 3) // 4)
    fft = 2.5 * ng * math.log2(ng)  # one real transform
    pairs = nb * (nb + 1)           # a multiply-add for each pair of bins
    node, part = ng * pairs, npart * (2.0 * sten * nb + pairs)
    forms = case.get("forms", "").split(",")
    per_lm = nb * fft + (node if "node" in forms else 0) + (node if "gamma" in forms else 0) + (part if "particle" in forms else 0)
    if kind in ("zeta", "batch"):
        cats = case.get("ncat", 1)
        return {"bytes": 16 * npart + 8 * cats * len(forms) * (case["lmax"] + 1) * nb * nb,
                "flops": cats * (fft + lm * (per_lm if kind == "zeta" else per_lm - (part if "particle" in forms else 0)))
                + (lm * part if kind == "batch" and "particle" in forms else 0)}
    if kind == "catalogue":
        return {"bytes": 32 * npart + 8 * ng + 8 * (n // 8) ** 3, "flops": fft + 2.0 * sten * npart}
    if kind == "fields":
        return {"bytes": 4 * ng + 4 * lanes * ng, "flops": nb * fft}
    if kind == "grid_sum":
        return {"bytes": 4 * ng + 4 * lanes * ng, "flops": node}
    if kind == "particle_sum":
        return {"bytes": 16 * npart + 4 * lanes * ng, "flops": part}
    if kind == "xi":
        return {"bytes": 16 * npart + 16 * nb, "flops": (nb + 1) * fft + 4.0 * sten * npart * nb}
    if kind == "grad_node":
        return {"bytes": 8 * ng, "flops": 2 * fft + lm * (2 * nb * fft + 2.0 * ng * nb * nb)}
    return {"bytes": 28 * npart, "flops": 2 * fft + lm * (2 * nb * fft + npart * nb * (8.0 * sten + 2.0 * nb))}


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind == "zeta":
        return _zeta(case, s["parts"])
    if kind == "batch":
        z = [_zeta(case, p) for p in s["parts"].split([int(v) for v in s["sizes"]])]
        return torch.stack([torch.stack([x[f] for f in FORMS if f in x]) for x in z])
    if kind == "catalogue":
        delta = _contrast(case, s["parts"])
        return {"delta": delta, "dhat": torch.view_as_real(_half(delta).contiguous()), "sorted": None, "start": None,
                "wsum": s["parts"][:, 3].double().sum().reshape(1)}
    if kind == "fields":
        dhat = torch.view_as_complex(s["dhat"]).to(torch.complex128)
        return _interleave(case, _fields(case, dhat, case["l"], case["m"], _radial(case, case["l"])), torch.float64)
    if kind in ("grid_sum", "particle_sum"):
        a = [s["alm"][b // 4, ..., b % 4].double() for b in range(case["nb"])]
        if kind == "particle_sum":
            f = _points(case, a, s["parts"])
            return (f * s["parts"][:, 3:].double()).T @ f / s["parts"][:, 3].double().sum()
        delta = s["delta"].double()
        if case["form"] == "gamma":
            return _gamma_sum(case, delta, a)
        v = torch.stack(a).reshape(case["nb"], -1)
        return torch.stack([(v * (delta.reshape(1, -1) * v[b])).sum(1) for b in range(case["nb"])]) / delta.numel()
    if kind == "xi":
        parts = s["parts"]
        delta = _contrast(case, parts)
        a = list(_fields(case, _half(delta), 0, 0, _radial(case, 0)))
        node = torch.stack([(x * delta).mean() for x in a])
        f = _points(case, a, parts)
        return {"node": node, "particle": (f * parts[:, 3:].double()).sum(0) / parts[:, 3].double().sum()}
    w = torch.from_numpy(s["weights"]).to("cuda")
    if kind == "grad_node":
        return _grad_node(case, s["delta"].double(), w)
    return _grad_particles(case, s["parts"], w)
