"""Workloads of the library as a user's program runs them, for timing and for comparing results.

A case is a dict of plain values; ``kind`` says which public entry points it goes through:

* ``recon``: ``pet.reconstruct``, f^0 to f^T with the objective history;
* ``iter``: a resident ``pet.State``, one outer iteration (every subset once) from f^0, then the
  image read back: the loop of a program that steps a scan itself;
* ``forward`` / ``back``: the stand-alone projectors over all views (simulation, normalisation);
* ``batch``: many scans of different sizes stepped together by ``pet.Batch``.

Inputs are seeded: phantoms of ``synth``, their analytic line integrals (evaluated here on the
GPU, never by the library), a uniform background of 10 % and Poisson counts.
"""
import math

import numpy as np
import torch

from paper_2111_07886_gb300 import pet, synth

# The workloads' SDP-P2 settings; f^0 = 1 everywhere, as a program without a prior image starts.
PARAMS = dict(beta=0.05, gamma_r=2.0, eps=1e-12, t=1e-4, U=1000.0, lambda0=1.0, a=0.45, rho=2.0,
              delta1=5.0, delta2=5.0, nu1=0.8, nu2=1.5, J0=3, J1=1000)
PRECOND = dict(bsrem=synth.PRECOND_BSREM, m1=synth.PRECOND_M1, m2=synth.PRECOND_M2,
               p1=synth.PRECOND_P1, p2=synth.PRECOND_P2)
PRECISION = dict(fp32=synth.PREC_FP32, kahan=synth.PREC_FP32_KAHAN, fp64=synth.PREC_FP64)


def _case(name, kind, n, planes, views, bins, subsets, **more):
    c = dict(name=name, kind=kind, n=n, planes=planes, views=views, bins=bins, subsets=subsets,
             pixel_mm=512.0 / max(n, 1), counts=1e6 * planes, iterations=1, precond="p2",
             precision="kahan", prior="rdp", beta=0.05, attn=False, subrays=1, ring_mm=0.0,
             bin_mm=0.0, tof_bins=0, tof_bin_mm=0.0, tof_fwhm_mm=0.0, scans=1, scan_seed=0)
    c.update(more)
    return c


def listed():
    return [
        # the plain 2-D method at its configured size: 120 subiterations of ~16 k pixels each,
        # a call made of many small launches
        _case("recon_2d_128", "recon", 128, 1, 180, 185, 12, iterations=10, pixel_mm=4.0),
        # the clinical-size stack, 20 iterations with the objective after each: the headline run
        _case("recon_stacked_256x89", "recon", 256, 89, 288, 357, 24, iterations=20, pixel_mm=2.7,
              beta=0.02, counts=5e7),
        # the smallest scan a program steps by itself (quick-look size): latency only
        _case("iter_2d_64", "iter", 64, 1, 60, 91, 6, precond="p1"),
        # a stack of odd sizes (planes not a multiple of the group, unequal subsets), plain FP32
        # sums
        _case("iter_stack_201x43", "iter", 201, 43, 211, 289, 17, precision="fp32", counts=4.3e7),
        # the paper's scanner: 576-detector ring, 32 rays per detector pair, attenuation
        _case("iter_ring_256", "iter", 256, 1, 288, 155, 24, pixel_mm=1.17, ring_mm=576 * 4.0 / (2 * math.pi),
              bin_mm=2.0, subrays=32, attn=True, counts=6.8e6, beta=0.1, precond="p1"),
        # the clinical stack as time-of-flight data
        _case("iter_tof_256x89", "iter", 256, 89, 288, 357, 24, pixel_mm=2.7, beta=0.02, counts=5e7,
              tof_bins=13, tof_bin_mm=60.0, tof_fwhm_mm=82.5),
        # the fully 3-D prior with per-bin detection factors: a clinical volume with attenuation
        _case("iter_rdp3d_attn_256x89", "iter", 256, 89, 288, 357, 24, pixel_mm=2.7, beta=0.02,
              counts=5e7, prior="rdp3d", attn=True),
        # the non-smooth prior: ten primal-dual steps after each subiteration
        _case("iter_tv_200x24", "iter", 200, 24, 240, 289, 24, prior="tv", counts=2e7),
        # the double-precision path of an accuracy study
        _case("iter_f64_128x16", "iter", 128, 16, 180, 185, 12, precision="fp64", pixel_mm=4.0,
              counts=8e6),
        # all-view projections of a stack: simulating data, and a plain backprojection
        _case("forward_256x89", "forward", 256, 89, 288, 357, 24, pixel_mm=2.7, counts=5e7),
        _case("back_256x89", "back", 256, 89, 288, 357, 24, pixel_mm=2.7, counts=5e7),
        # 2-D scans of different sizes, views and subsets advanced together (batched serving)
        _case("batch_mixed_24", "batch", 0, 1, 0, 0, 0, scans=24, iterations=10, scan_seed=1),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: 2-D scans of 64^2..400^2, stacks of 2..89 planes, every
    option of the listed ones."""
    what = rng.choice(["recon2d", "reconstack", "iter2d", "iterstack", "iterstack", "ring", "tof", "rdp3d",
                       "tv", "f64", "forward", "back", "batch"])
    counts = math.exp(rng.uniform(math.log(1e6), math.log(1e7)))
    if what == "batch":
        return _draw_clean(_case("", "batch", 0, 1, 0, 0, 0, scans=rng.randint(3, 24), iterations=rng.randint(2, 10),
                                 scan_seed=rng.randint(2, 10 ** 6)))
    flat = what in ("recon2d", "iter2d", "ring")
    n = _logint(rng, 64, 400 if what in ("recon2d", "iter2d") else 256)
    views = rng.randint(60, 288)
    bins = max(4, int(1.45 * n) - rng.randint(0, 6))
    subsets = rng.randint(4, min(36, views // 4))
    planes = 1 if flat else _logint(rng, 2, 89)
    # Nesterov's alpha (up to 2) over many subsets of noisy data lets rounding grow: few subsets there
    more = dict(counts=counts * planes, precond=rng.choice(["p1", "m1", "p2"] if subsets <= 8 else ["p2", "p2", "m2", "bsrem"]),
                precision=rng.choice(["kahan", "kahan", "fp32"]))
    kind = "iter"
    if what == "recon2d":
        kind, more["iterations"] = "recon", rng.randint(2, 12)
    elif what == "reconstack":
        kind, more["iterations"] = "recon", rng.randint(2, 10)
    elif what == "iterstack":
        more["attn"] = rng.random() < 0.3
    elif what == "ring":
        n = _logint(rng, 128, 256)
        more.update(pixel_mm=300.0 / n, ring_mm=576 * 4.0 / (2 * math.pi), bin_mm=2.0, subrays=rng.choice([1, 8, 17, 32]),
                    attn=rng.random() < 0.7)
        bins = 155
    elif what == "tof":
        n, planes = _logint(rng, 64, 200), _logint(rng, 1, 48)
        bins = max(4, int(1.45 * n) - rng.randint(0, 6))
        more.update(counts=counts * planes, tof_bins=rng.randint(7, 21), tof_bin_mm=rng.uniform(30.0, 70.0),
                    tof_fwhm_mm=rng.uniform(50.0, 100.0))
    elif what == "rdp3d":
        more.update(prior="rdp3d", attn=rng.random() < 0.5)
    elif what == "tv":
        n, planes = _logint(rng, 64, 256), _logint(rng, 1, 32)
        bins = max(4, int(1.45 * n) - rng.randint(0, 6))
        more.update(prior="tv", counts=counts * planes)
    elif what == "f64":
        n, planes = _logint(rng, 48, 128), _logint(rng, 1, 24)
        bins = max(4, int(1.45 * n) - rng.randint(0, 6))
        more.update(precision="fp64", counts=counts * planes)
    elif what in ("forward", "back"):
        kind = what
    return _draw_clean(_case("", kind, n, planes, views, bins, subsets, **more))


def _draw_clean(c):
    del c["name"]
    return c


def _mixed(case):
    """The scans of a batch case, each a case of its own: the sizes of mixed 2-D studies with 1e6 to
    1e7 counts (with fewer, a scan's iterates amplify rounding and no two programs agree on them)."""
    out = []
    for w in synth.mixed_2d_scans(case["scans"], case["scan_seed"], case["iterations"]):
        out.append(_case("", "recon", w.n, 1, w.nviews, w.nbins, w.nsubsets, iterations=case["iterations"],
                         pixel_mm=w.pixel_mm, counts=1e6 * math.sqrt(w.counts / 1e5)))
    return out


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

def _bin_mm(c):
    return c["bin_mm"] or c["pixel_mm"]


def _angles(c):
    th = [v * math.pi / c["views"] for v in range(c["views"])]
    return torch.tensor(th, dtype=torch.float64, device="cuda")


def _offsets(c):
    """Bin centres in mm."""
    k = torch.arange(c["bins"], dtype=torch.float64, device="cuda") - 0.5 * (c["bins"] - 1)
    return c["ring_mm"] * torch.sin(k * _bin_mm(c) / c["ring_mm"]) if c["ring_mm"] else k * _bin_mm(c)


def _inputs(c, seed):
    """counts (int32), gamma and the detection factors (float32, [P][V][NB] or [P][V][NB][T]),
    and sens, for the analytic projections of a seeded phantom."""
    n, planes = c["n"], c["planes"]
    if planes == 1:
        shapes = synth.ellipse_phantom_2d(n, c["pixel_mm"], seed)
    else:
        shapes = synth.ellipsoid_phantom_3d(n, planes, c["pixel_mm"], c["pixel_mm"], seed)
    most = max(len(s) for s in shapes)
    rows = [list(s) + [(0.0, 0.0, 1.0, 1.0, 0.0, 0.0)] * (most - len(s)) for s in shapes]
    e = torch.tensor(rows, dtype=torch.float32, device="cuda")             # [P][shapes][6]
    th, r = _angles(c).float()[None, :, None], _offsets(c).float()[None, None, :]
    tof = c["tof_bins"] if c["tof_bins"] > 1 else 0
    full = (planes, c["views"], c["bins"]) + ((tof,) if tof else ())
    sino = torch.zeros(full, device="cuda")
    body = None
    sig = c["tof_fwhm_mm"] / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    edges = [(t - tof / 2.0) * c["tof_bin_mm"] for t in range(tof + 1)]
    for k in range(most):
        cx, cy, a, b, phi, val = (e[:, k, q][:, None, None] for q in range(6))
        d2 = (a * torch.cos(th - phi)) ** 2 + (b * torch.sin(th - phi)) ** 2
        rp = r - (cx * torch.cos(th) + cy * torch.sin(th))
        chord = 2.0 * a * b * torch.sqrt((d2 - rp * rp).clamp_min(0.0)) / d2
        if k == 0 and c["attn"]:
            body = chord * (val != 0)
        if not tof:
            sino += val * chord
            continue
        # the chord's middle along the line (-sin, cos), then each TOF bin's Gaussian share
        mid = (-cx * torch.sin(th) + cy * torch.cos(th)) \
            + rp * (b * b - a * a) * torch.sin(th - phi) * torch.cos(th - phi) / d2
        last = None
        for t, edge in enumerate(edges):
            z1, z2 = (edge - mid + 0.5 * chord) / sig, (edge - mid - 0.5 * chord) / sig
            psi = [z * torch.special.ndtr(z) + torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi) for z in (z1, z2)]
            f = sig * (psi[0] - psi[1])
            if last is not None:
                sino[..., t - 1] += val * (f - last).clamp_min(0.0)
            last = f
    mult = None
    if c["attn"]:
        mult = torch.exp(-synth.PAPER_MU_WATER_PER_MM * body)
        mult = (mult[..., None].expand(full) if tof else mult).contiguous()
        sino *= mult
    total = float(sino.sum(dtype=torch.float64))
    sens = c["counts"] / (1.1 * total)
    gamma = torch.full(full, 0.1 * sens * total / sino.numel(), device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    counts = torch.poisson(sino.mul_(sens).add_(gamma), generator=g).to(torch.int32)
    return counts, gamma, mult, sens


def _params(c):
    p = synth.AlgoParams(iterations=c["iterations"], precond=PRECOND[c["precond"]], **dict(PARAMS, beta=c["beta"]))
    p.precision = PRECISION[c["precision"]]
    p.rdp3d = int(c["prior"] == "rdp3d")
    p.reg = int(c["prior"] == "tv")
    return p


def _geometry(c, sens):
    return pet.Geometry(c["n"], c["planes"], c["pixel_mm"], c["views"], c["bins"], _bin_mm(c), c["subsets"], sens,
                        subrays=c["subrays"], tof_bins=c["tof_bins"], tof_bin_mm=c["tof_bin_mm"],
                        tof_fwhm_mm=c["tof_fwhm_mm"], ring_mm=c["ring_mm"])


def _ones(c):
    return torch.ones((c["planes"], c["n"], c["n"]), device="cuda")


def _field(c, shape, seed):
    """A positive, uneven float32 field: the operand of a stand-alone projector."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(shape, generator=g, device="cuda") * 1.9 + 0.1


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        stream, scans = torch.cuda.Stream(), []
        for k, m in enumerate(_mixed(c)):
            counts, gamma, _, sens = _inputs(m, seed + 7919 * k)
            g = _geometry(m, sens)
            s = pet.State(g, counts, gamma, pet.make_params(_params(m)), _ones(m))
            scans.append((g, s, torch.empty((1, m["n"], m["n"]), device="cuda")))
        torch.cuda.synchronize()
        return dict(case=c, scans=scans, batch=pet.Batch(len(scans)), stream=stream)
    if c["kind"] in ("forward", "back"):
        g = _geometry(c, 0.01)
        img, proj = (c["planes"], c["n"], c["n"]), (c["planes"], c["views"], c["bins"])
        src, dst = (img, proj) if c["kind"] == "forward" else (proj, img)
        return dict(case=c, g=g, src=_field(c, src, seed), dst=torch.empty(dst, device="cuda"))
    counts, gamma, mult, sens = _inputs(c, seed)
    g, p = _geometry(c, sens), pet.make_params(_params(c))
    st = dict(case=c, g=g, params=p, init=_ones(c))
    if c["kind"] == "recon":
        return dict(st, counts=counts, gamma=gamma, img=torch.empty_like(st["init"]))
    st["state"] = pet.State(g, counts, gamma, p, st["init"], d_mult=mult)
    wide = torch.float64 if c["precision"] == "fp64" else torch.float32
    st["out"] = torch.empty(st["init"].shape, dtype=wide, device="cuda")
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "recon":
        state["img"].copy_(state["init"])
        phi = pet.reconstruct(state["g"], state["counts"], state["gamma"], state["params"], state["img"], objective=True)
        return {"image": state["img"], "objective": np.asarray(phi, np.float32)}
    if c["kind"] == "iter":
        s = state["state"]
        s.reset(state["init"])
        for _ in range(c["subsets"]):
            s.subiter()
        s.read_image(state["out"])
        return state["out"]
    if c["kind"] == "forward":
        pet.forward_subset(state["g"], -1, state["src"], state["dst"])
        return state["dst"]
    if c["kind"] == "back":
        pet.back_subset(state["g"], -1, state["src"], state["dst"])
        return state["dst"]
    b, stream = state["batch"], state["stream"]
    for _, s, _ in state["scans"]:
        if s in b.members:
            b.remove(s)
        s.reset(stream=stream)
    for _, s, _ in state["scans"]:
        b.add(s, with_objective=True, stream=stream)
    while b.step(stream=stream) > 0:
        pass
    for _, s, out in state["scans"]:
        s.read_image(out, stream=stream)
    return {"images": [out for _, _, out in state["scans"]],
            "objective": [np.asarray(s.objective_history(stream=stream), np.float32) for _, s, _ in state["scans"]]}


def work(case):
    """Bytes: each input read and each output written once.  Operations: a multiply-add for every
    (line, pixel, plane) crossing of each projection and backprojection (a view's lines cross
    n^2 4/pi pixels per pixel of line spacing on average), and about 100 per voxel and
    subiteration for the prior and the step."""
    c = case
    if c["kind"] == "batch":
        parts = [work(m) for m in _mixed(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    q = c["planes"] * c["n"] ** 2
    tof = max(1, c["tof_bins"])
    sino = c["planes"] * c["views"] * c["bins"] * tof
    spacing = _bin_mm(c) / c["pixel_mm"]
    cover = min(1.0, (c["bins"] * spacing / c["n"]))
    proj = 2.0 * 4.0 / math.pi * q * c["views"] * c["subrays"] * tof / spacing * cover
    if c["kind"] in ("forward", "back"):
        return {"bytes": 4.0 * (q + sino), "flops": proj}
    steps = c["iterations"] if c["kind"] == "recon" else 1
    flops = steps * (2.0 * proj + 100.0 * q * c["subsets"])
    if c["prior"] == "tv":
        flops += 10 * 20.0 * q * c["subsets"] * steps
    if c["kind"] == "recon":
        flops += (steps + 1) * proj
    return {"bytes": 4.0 * (2 * q + (3 if c["attn"] else 2) * sino), "flops": flops}


# ------------------------------------------------------------------------------------------
# The same results in 64 bits, from the equations: the system matrix of each subset as a sparse
# matrix (each line cut at the pixel columns, or rows, of the axis it follows), the Table I loop
# ------------------------------------------------------------------------------------------

def _matrix(c, views):
    """A of these views (rows [view][bin][tof]) and its transpose, without sens, as sparse CSR."""
    n, nb, dev = c["n"], c["bins"], "cuda"
    rho, sub = _bin_mm(c) / c["pixel_mm"], c["subrays"]
    tof = max(1, c["tof_bins"])
    k = torch.arange(nb, dtype=torch.float64, device=dev) - 0.5 * (nb - 1)
    if c["ring_mm"]:
        rd, db = c["ring_mm"] / c["pixel_mm"], _bin_mm(c) / c["ring_mm"]
        lo, hi, centre = rd * torch.sin((k - 0.5) * db), rd * torch.sin((k + 0.5) * db), rd * torch.sin(k * db)
    else:
        centre, lo, hi = k * rho, (k - 0.5) * rho, (k + 0.5) * rho
    if sub > 1:
        part = (torch.arange(sub, dtype=torch.float64, device=dev) + 0.5) / sub
        lines = lo[:, None] + (hi - lo)[:, None] * part[None, :]           # [bin][line]
    else:
        lines = centre[:, None]
    d = torch.arange(n, dtype=torch.float64, device=dev)
    rows, cols, vals = [], [], []
    for u, v in enumerate(views):
        th = v * math.pi / c["views"]
        co, si = math.cos(th), math.sin(th)
        co, si = (0.0 if abs(co) < 1e-12 else co), (0.0 if abs(si) < 1e-12 else si)
        along_x = abs(si) >= abs(co)
        big, small = (si, co) if along_x else (co, si)
        # cross coordinate (grid units) where the line enters and leaves each step d
        x0 = lines[..., None] / big + 0.5 * n * (1.0 + small / big) - (small / big) * d
        a = x0 + min(0.0, -small / big)
        b = x0 + max(0.0, -small / big)
        ra, rb = torch.floor(a), torch.floor(b)
        cross = rb != ra
        far = torch.where(cross, (b - rb) / (abs(small) if small else 1.0), torch.zeros_like(b))
        near = 1.0 / abs(big) - far
        row = (u * nb + torch.arange(nb, device=dev))[:, None, None].expand_as(a)
        step = d.long().expand_as(a)
        for r, length, on in ((ra, near, ra == ra), (rb, far, cross)):
            on = on & (r >= 0) & (r < n)
            rr, dd = r[on].long(), step[on]
            rows.append(row[on])
            cols.append(rr * n + dd if along_x else dd * n + rr)
            vals.append(length[on] / sub)
    rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    if tof > 1:
        sig = c["tof_fwhm_mm"] / (2.0 * math.sqrt(2.0 * math.log(2.0))) / c["pixel_mm"]
        w = c["tof_bin_mm"] / c["pixel_mm"]
        th = _angles(c)[torch.tensor(views, device=dev)][rows // nb]
        x, y = (cols % n) + 0.5 - 0.5 * n, torch.div(cols, n, rounding_mode="floor") + 0.5 - 0.5 * n
        tau = -x * torch.sin(th) + y * torch.cos(th)
        out = []
        for t in range(tof):
            z0, z1 = ((t - tof / 2.0) * w - tau) / sig, ((t + 1 - tof / 2.0) * w - tau) / sig
            flip = z0 > 0
            h = torch.special.ndtr(torch.where(flip, -z0, z1)) - torch.special.ndtr(torch.where(flip, -z1, z0))
            on = h > 1e-18
            out.append((rows[on] * tof + t, cols[on], vals[on] * h[on]))
        rows, cols, vals = (torch.cat([o[q] for o in out]) for q in range(3))
    size = (len(views) * nb * tof, n * n)

    def csr(i, j, shape):
        key, order = torch.sort(i * shape[1] + j)
        key, count = torch.unique_consecutive(key, return_counts=True)
        v = torch.zeros(key.numel(), dtype=torch.float64, device=dev)
        v.index_add_(0, torch.repeat_interleave(torch.arange(key.numel(), device=dev), count), vals[order])
        r = torch.div(key, shape[1], rounding_mode="floor")
        ptr = torch.zeros(shape[0] + 1, dtype=torch.int64, device=dev)
        ptr[1:] = torch.cumsum(torch.bincount(r, minlength=shape[0]), 0)
        return torch.sparse_csr_tensor(ptr, key % shape[1], v, shape)

    return csr(rows, cols, size), csr(cols, rows, (size[1], size[0]))


def _rdp(f, three_d, gamma_r, eps):
    """(gradient, value) of the relative difference prior; f [P][N][N]."""
    grad, value = torch.zeros_like(f), 0.0
    P, n, _ = f.shape
    for dz in ((-1, 0, 1) if three_d else (0,)):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if not (dz or dy or dx):
                    continue
                def cut(d, m):
                    return slice(max(0, -d), m - max(0, d)), slice(max(0, d), m + min(0, d))
                (z0, z1), (y0, y1), (x0, x1) = cut(dz, P), cut(dy, n), cut(dx, n)
                if P <= abs(dz):
                    continue
                j, k = f[z0, y0, x0], f[z1, y1, x1]
                diff = j - k
                den = j + k + gamma_r * diff.abs() + eps
                value += float((diff * diff / den).sum())
                grad[z0, y0, x0] += 2.0 * diff * (gamma_r * diff.abs() + j + 3.0 * k + 2.0 * eps) / (den * den)
    return grad, value


def _slope(f, dim):
    """Matlab's gradient along one axis: central inside, one-sided at the ends."""
    m = f.shape[dim]
    if m == 1:
        return torch.zeros_like(f)
    up = torch.cat([f.narrow(dim, 1, m - 1), f.narrow(dim, m - 1, 1)], dim)
    dn = torch.cat([f.narrow(dim, 0, 1), f.narrow(dim, 0, m - 1)], dim)
    h = torch.full((m,), 0.5, dtype=f.dtype, device=f.device)
    h[0] = h[-1] = 1.0
    return (up - dn) * h.view([-1 if q == dim else 1 for q in range(3)])


def _tv_prox(z, w, b, p, iters):
    """Primal-dual steps from x = z; p: the dual variable, updated in place."""
    x, xbar, tau = z, z, 0.25 / b
    for _ in range(iters):
        gx, gy = torch.zeros_like(z), torch.zeros_like(z)
        gx[..., :-1] = xbar[..., 1:] - xbar[..., :-1]
        gy[:, :-1] = xbar[:, 1:] - xbar[:, :-1]
        qx, qy = p[0] + 0.5 * gx, p[1] + 0.5 * gy
        s = torch.sqrt(qx * qx + qy * qy).clamp_min(1.0)
        p[0], p[1] = qx / s, qy / s
        div = p[0] + p[1]
        div[..., 1:] -= p[0][..., :-1]
        div[:, 1:] -= p[1][:, :-1]
        r = tau / w
        xn = (x + 0.25 * div + r * z) / (1.0 + r)
        xbar, x = 2.0 * xn - x, xn
    return x


def _reconstruct64(c, counts, gamma, mult, sens, objective):
    """f^T and Phi(f^k) in 64 bits (Table I), from f^0 = 1."""
    n, P, M, p = c["n"], c["planes"], c["subsets"], dict(PARAMS, beta=c["beta"])
    scale = sens * c["pixel_mm"]

    def flat(t, views):                        # [P][V].. -> [rows][P] of these views
        t = t.reshape(P, c["views"], -1)[:, views].reshape(P, -1)
        return t.t().double().contiguous()

    subs = []
    for i in range(M):
        views = list(range(i, c["views"], M))
        A, At = _matrix(c, views)
        subs.append((A, At, flat(counts, views), flat(gamma, views), None if mult is None else flat(mult, views)))
    pj = torch.zeros((n * n, P), dtype=torch.float64, device="cuda")
    for A, At, g, _, m in subs:
        pj += scale * (At @ (torch.ones_like(g) if m is None else m))
    pj = torch.where(pj > 0, pj / M, torch.full_like(pj, 1.0 / M)).t().reshape(P, n, n)
    f = torch.ones((P, n, n), dtype=torch.float64, device="cuda")
    dual = [torch.zeros_like(f), torch.zeros_like(f)]
    three, phis, tn = c["prior"] == "rdp3d", [], 1.0

    def mean_data(A, f, gam, m):
        y = scale * (A @ f.reshape(P, -1).t().contiguous())
        return y if m is None else m * y

    def phi():
        v = 0.0
        for A, _, g, gam, m in subs:
            y = mean_data(A, f, gam, m)
            v += float(y.sum()) - float(torch.where(g > 0, g * torch.log(y + gam), torch.zeros_like(g)).sum())
        return v + p["beta"] * _rdp(f, three, p["gamma_r"], p["eps"])[1]

    if objective:
        phis.append(phi())
    for k in range(c["iterations"]):
        for i in range(M):
            J = k * M + i + 1
            lam, alpha = p["lambda0"] / (p["a"] * k + 1.0), 1.0
            if c["precond"] in ("m1", "p1"):
                t1 = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * tn * tn))
                alpha, tn = 1.0 + (tn - 1.0) / t1, t1
            elif c["precond"] in ("m2", "p2"):
                alpha = (p["rho"] * (J - 1) + p["delta2"]) / ((J - 1) + p["delta1"])
            nu = torch.ones_like(f)
            if c["precond"] in ("p1", "p2") and p["J0"] < J <= p["J1"]:
                sq = _slope(f, 2) ** 2 + _slope(f, 1) ** 2 + (_slope(f, 0) ** 2 if three else 0.0)
                mu = (torch.sqrt(sq) / f.mean()).clamp_min(0.01)
                nu = (mu.mean() / mu).clamp(p["nu1"], p["nu2"])
            A, At, g, gam, m = subs[i]
            ratio = 1.0 - g / (mean_data(A, f, gam, m) + gam)
            grad = scale * (At @ (ratio if m is None else m * ratio)).t().reshape(P, n, n)
            step = lam * alpha * nu * torch.where(f < 0.5 * p["U"], f, p["U"] - f) / pj
            if c["prior"] == "tv":
                f = _tv_prox(f - step * grad, step, p["beta"] / M, dual, 10)
            else:
                f = f - step * (grad + p["beta"] / M * _rdp(f, three, p["gamma_r"], p["eps"])[0])
            f = torch.where(f <= 0, torch.full_like(f, p["t"]), torch.where(f >= p["U"], torch.full_like(f, p["U"] - p["t"]), f))
        if objective:
            phis.append(phi())
    return f, phis


def exact(case, seed):
    c = case
    if c["kind"] in ("forward", "back"):
        img, proj = (c["planes"], c["n"], c["n"]), (c["planes"], c["views"], c["bins"])
        src = _field(c, img if c["kind"] == "forward" else proj, seed).double()
        scale, flat = 0.01 * c["pixel_mm"], src.reshape(c["planes"], -1).t().contiguous()
        out = torch.zeros((c["views"] * c["bins"] if c["kind"] == "forward" else c["n"] ** 2, c["planes"]),
                          dtype=torch.float64, device="cuda")
        for v0 in range(0, c["views"], 16):
            views = list(range(v0, min(c["views"], v0 + 16)))
            rows = slice(v0 * c["bins"], (v0 + len(views)) * c["bins"])
            A, At = _matrix(c, views)
            if c["kind"] == "forward":
                out[rows] = A @ flat
            else:
                out += At @ flat[rows]
        return (scale * out).t().reshape(proj if c["kind"] == "forward" else img)
    if c["kind"] == "batch":
        images, phis = [], []
        for k, m in enumerate(_mixed(c)):
            f, phi = _reconstruct64(m, *_inputs(m, seed + 7919 * k), True)
            images.append(f)
            phis.append(np.asarray(phi))
        return {"images": images, "objective": phis}
    f, phi = _reconstruct64(c, *_inputs(c, seed), c["kind"] == "recon")
    return {"image": f, "objective": np.asarray(phi)} if c["kind"] == "recon" else f
