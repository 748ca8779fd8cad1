"""Performance cases: what a program that uses this package has it do, through its public calls.

The specimens are those of this repository's configurations: rocksalt Fe-O crystals
(a = 4.3 A, slices of a/2) and an Fe-O sphere of 80 A in a 100 A box (slices of 2 A), with
two-Gaussian projected potentials, 200 keV, a 20 mrad probe and a 30 mrad EELS aperture,
and synthetic L-edge transition potentials on every Fe atom.  Every atom is displaced by a
seeded Gaussian offset (0.08 A, one frozen-phonon configuration), so that each seed is
another specimen; potentials, window origins and transition potentials follow the displaced
atoms.  Results are returned as the calls give them: complex64 S-matrices, FP64 maps.

Kinds of case
  map      the S-matrix is kept by the program, one EELS map per pass
  request  build of the S-matrix and the map from it
  phonon   the frozen-phonon average: build and map of two configurations
  build    the S-matrix at every depth, copied into the program's tensor
  elastic  ADF and incoherent bright-field images from a kept S-matrix
  serve    requests of uneven sizes on the map server, host arrays in, host maps out
"""
import math

import numpy as np
import torch

import paper_1908_07628_gb300 as eels

A = 4.3                    # lattice constant, A
LAM, SIGMA = 0.02508, 7.2886e-4
ALPHA, BETA = 0.020, 0.030
POTENTIAL = (((80.0, 0.25), (20.0, 0.8)), ((30.0, 0.25), (8.0, 0.8)))   # Fe, O: (V A, A)
M_ORDER = (0, 1, -1, 2, -2, 3)
DETECTORS = ((0.060, 0.0), (0.0, BETA))


def _case(name, kind, n, cell, n_z, f, w=0, types=0, nsx=0, nsy=0, precision="", grouping="model",
          shared=False, sphere=0.0):
    return {"name": name, "kind": kind, "n": n, "cell": cell, "n_z": n_z, "f": f, "w": w,
            "types": types, "nsx": nsx, "nsy": nsy, "precision": precision, "grouping": grouping,
            "shared": shared, "sphere": sphere}


def listed():
    return [
        # the smallest call: a few probes over a thin crystal of one cell, default precision;
        # launches, allocations and host work are all there is
        _case("map_tiny_fp32", "map", 64, A, 4, 1, 13, 2, 3, 3, "fp32"),
        # the check-out size: one 2 x 2 cell crystal, whole cell imaged, default precision
        _case("request_small_fp32", "request", 128, 2 * A, 6, 1, 32, 3, 8, 8, "fp32"),
        # frozen-phonon averaging in the default precision (CUDA-core contraction)
        _case("phonon_256_fp32", "phonon", 256, 4 * A, 12, 2, 24, 3, 16, 16, "fp32"),
        # a thickness-series slab on a coarse grid, small scan, TF32 split
        _case("slab_256_tf32", "map", 256, 8 * A, 12, 2, 32, 3, 16, 16, "tf32"),
        # a dense ragged scan with one channel: many probes per site, so the transition is
        # contracted first; a grid with a factor of three
        _case("dense_384_bf16", "map", 384, 6 * A, 16, 3, 21, 1, 61, 67, "bf16x3"),
        # the 8 x 8 cell crystal at its full grid and scan, TF32 split
        _case("crystal_512_tf32", "map", 512, 8 * A, 8, 2, 32, 3, 32, 32, "tf32"),
        # S-matrix build, grid with a factor of three, f = 3
        _case("build_768", "build", 768, 12 * A, 6, 3),
        # the 12 x 12 cell crystal, BF16 split
        _case("crystal_768_bf16", "map", 768, 12 * A, 10, 2, 32, 3, 32, 32, "bf16x3"),
        # S-matrix build on the largest grid
        _case("build_1024", "build", 1024, 100.0, 5, 4, sphere=80.0),
        # the central slices of the 80 A sphere, 128 x 128 scan, the library's own grouping
        _case("sphere_1024_bf16", "map", 1024, 100.0, 8, 4, 24, 3, 128, 128, "bf16x3", "auto",
              sphere=80.0),
        # ADF and bright-field images of the 8 x 8 cell crystal
        _case("elastic_512", "elastic", 512, 8 * A, 4, 2, nsx=32, nsy=32),
        # the map server: six requests of uneven sizes at once (see _requests)
        _case("serve_mixed", "serve", 512, 8 * A, 16, 3, 32, 3, 24, 24, "bf16x3", shared=True),
    ]


def draw(rng):
    """A case of the listed ranges: every kind, grid, f, precision; thickness, windows and
    scans spread over their range, odd and non-square ones among them."""
    def spread(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5)))))))

    top = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("map", "map", "map", "request", "phonon", "build", "elastic", "serve"))
        n = rng.choice((64, 128, 256, 384, 512, 768, 1024))
        f = rng.choice((1, 2, 3, 4))
        sphere = 80.0 if kind in ("map", "build") and n == 1024 and rng.random() < 0.5 else 0.0
        if sphere:
            cell, n_z, f = 100.0, spread(2, 8), 4
        else:
            cells = max(1, n // rng.choice((32, 64, 64)))
            cell, n_z = cells * A, spread(3, 40)
        c = _case("", kind, n, cell, n_z, f, spread(8, 32), rng.randint(1, 6), spread(2, 64),
                  spread(2, 64), rng.choice(("fp32", "tf32", "bf16x3", "bf16x3")), "model",
                  rng.random() < 0.5, sphere)
        if kind in ("build", "elastic"):
            c.update(w=0, types=0, precision="", shared=False)
        if kind == "build":
            c.update(nsx=0, nsy=0)
        if kind == "serve":
            c.update(n=rng.choice((256, 384, 512)), precision=rng.choice(("tf32", "bf16x3")),
                     shared=True)
            c["cell"] = c["n"] // 64 * A
            c["f"] = rng.choice((2, 3, 4))
        if kind == "elastic" and (n < 64 * f or (n // 2) % f):
            continue
        if c["w"] > c["n"] // 2 or not _usable(c):
            continue
        if 1e-4 * top < _cost(c) <= top and _s_in_bytes(c) < 2.2e10:
            del c["name"]
            return c


# --- specimens ---------------------------------------------------------------------------

def _layers(c, rng):
    """Per slice: displaced atom positions (x, y) and whether each atom is Fe."""
    out = []
    if c["sphere"]:
        # lattice points inside the sphere, an Fe at the centre; the slices nearest the centre
        box, r = c["cell"], c["sphere"] / 2
        m = int(r / A) + 2
        g = np.arange(-m, m + 1)
        k, j, i = (v.ravel() for v in np.meshgrid(g, g, g, indexing="ij"))
        pts = []
        for fx, fy, fz in ((0, 0, 0), (.5, .5, 0), (.5, 0, .5), (0, .5, .5)):
            for fe in (True, False):
                p = np.stack([i + fx + (0 if fe else .5), j + fy, k + fz], 1) * A
                p = p[(p * p).sum(1) <= r * r]
                pts.append((p, np.full(len(p), fe)))
        p = np.concatenate([q for q, _ in pts])
        fe = np.concatenate([q for _, q in pts])
        sl = np.floor(p[:, 2] / 2.0 + 1e-9).astype(np.int64) + c["n_z"] // 2
        for s in range(c["n_z"]):
            q = p[sl == s][:, :2] + box / 2
            out.append((q + rng.normal(0, 0.08, q.shape), fe[sl == s]))
        return out, 2.0
    cells = int(round(c["cell"] / A))
    jj, ii = (v.ravel() for v in np.meshgrid(np.arange(cells), np.arange(cells), indexing="ij"))
    for s in range(c["n_z"]):
        fe_xy = ((0, 0), (.5, .5)) if s % 2 == 0 else ((.5, 0), (0, .5))
        ox_xy = ((.5, 0), (0, .5)) if s % 2 == 0 else ((0, 0), (.5, .5))
        q = [np.stack([ii + fx, jj + fy], 1) * A for fx, fy in fe_xy + ox_xy]
        fe = np.repeat([True, True, False, False], cells * cells)
        q = np.concatenate(q)
        out.append(((q + rng.normal(0, 0.08, q.shape)) % c["cell"], fe))
    return out, A / 2


def _potentials(c, layers):
    """Projected potentials [n_z][n][n] on the GPU: sums of periodic Gaussians, one product
    of row and column factors per slice."""
    n, cell = c["n"], c["cell"]
    grid = torch.arange(n, device="cuda", dtype=torch.float64) * (cell / n)
    v = torch.zeros((len(layers), n, n), device="cuda")
    for s, (xy, fe) in enumerate(layers):
        if not len(xy):
            continue
        d = grid[None, :, None] - torch.from_numpy(np.ascontiguousarray(xy)).cuda()[:, None, :]
        d = d - cell * torch.floor(d / cell + 0.5)
        amp = torch.tensor([[POTENTIAL[0 if x else 1][k][0] for x in fe] for k in (0, 1)],
                           device="cuda", dtype=torch.float64)
        for k, width in enumerate((0.25, 0.8)):
            g = torch.exp(-d * d / (2 * width * width))
            v[s] += ((g[:, :, 1] * amp[k][:, None]).t() @ g[:, :, 0]).float()
    return v


def _inputs(c, rng):
    """Everything one map takes: vproj and H on the GPU, site lists on the host."""
    layers, dz = _layers(c, rng)
    n, w, nh = c["n"], c["w"], c["n"] // 2
    px = c["cell"] / nh
    s = {"vproj": _potentials(c, layers), "dz": dz, "scan": _scan(c) if c["nsx"] else None}
    if not w:
        return s
    sites = [xy[fe] for xy, fe in layers]
    pos = np.concatenate(sites)
    near = np.floor(pos / px + 0.5).astype(np.int64)
    s["slice"] = np.repeat(np.arange(len(sites)), [len(q) for q in sites]).astype(np.int32)
    s["x"], s["y"] = (np.ascontiguousarray(pos[:, k]) for k in (0, 1))
    s["wx"], s["wy"] = (((near[:, k] - w // 2) % nh).astype(np.int32) for k in (0, 1))
    u = torch.arange(w, device="cuda", dtype=torch.float64)
    off = np.zeros((1, 2)) if c["shared"] else near * px - pos   # nearest pixel - site
    off = torch.from_numpy(off).cuda()
    dx = off[:, :1] + (u - w // 2)[None, :] * px
    dy = off[:, 1:] + (u - w // 2)[None, :] * px
    h = torch.empty((len(off), c["types"], w, w), dtype=torch.complex64, device="cuda")
    env = 0.01 * torch.exp(-(dx[:, None, :] ** 2 + dy[:, :, None] ** 2) / 0.18)
    for t, m in enumerate(M_ORDER[:c["types"]]):
        arm = torch.complex(dx[:, None, :].expand_as(env) / 0.3,
                            (1 if m >= 0 else -1) * dy[:, :, None].expand_as(env) / 0.3)
        h[:, t] = (env * arm ** abs(m)).to(torch.complex64)
    s["H"] = h[0].contiguous() if c["shared"] else h
    return s


def _scan(c):
    nsx, nsy = c["nsx"], c["nsy"]
    if c["sphere"]:
        return (nsx, nsy, 10.0, 10.0, 80.0 / nsx, 80.0 / nsy)
    c0 = int(round(c["cell"] / A)) // 2 * A
    return (nsx, nsy, c0, c0, A / nsx, A / nsy)


def _requests(c):
    """The serve cases' requests: uneven grids, thicknesses, channels and scans up to the
    case's own."""
    grids = [g for g in (256, 384, 512) if g <= c["n"]]
    out = []
    for k in range(6):
        n = grids[(k + len(grids) - 1) % len(grids)]
        out.append(dict(c, kind="request", n=n, cell=n // 64 * A,
                        n_z=max(2, c["n_z"] * (6 - k) // 6), types=1 + (c["types"] - 1) * k // 5,
                        nsx=max(2, c["nsx"] * (k + 3) // 8), nsy=max(2, c["nsy"] * (8 - k) // 8)))
    return out


def _configurations(c):
    if c["kind"] == "serve":
        return _requests(c)
    return [c, c] if c["kind"] == "phonon" else [c]


class _Workload:
    """A configuration with the attribute names that phonon_map unpacks."""

    def __init__(self, c, s):
        self.n, self.n_z, self.cell, self.f, self.dz = c["n"], c["n_z"], c["cell"], c["f"], s["dz"]
        self.lam, self.sigma, self.alpha, self.beta = LAM, SIGMA, ALPHA, BETA
        self.vproj, self.H, self.scan = s["vproj"], s["H"], s["scan"]
        self.site_slice, self.site_x, self.site_y = s["slice"], s["x"], s["y"]
        self.win_x0, self.win_y0 = s["wx"], s["wy"]


# --- the calls ---------------------------------------------------------------------------

def _optics(c, s):
    return (c["cell"], LAM, SIGMA, s["dz"], c["f"], ALPHA)


def _transitions(s):
    return (s["H"], s["slice"], s["wx"], s["wy"], s["x"], s["y"], s["scan"], BETA)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    sets = [_inputs(c, rng) for c in _configurations(case)]
    s = sets[0]
    state = {"case": case, "in": sets}
    if kind == "serve":
        # a program of the server has its requests in host memory
        state["server"] = eels.Server(0, hbm_budget=64 << 30, slots=4)
        state["requests"] = []
        for c, t in zip(_requests(case), sets):
            req, keep = eels.make_request(t["vproj"].cpu().numpy(), *_optics(c, t),
                                          t["H"].cpu().numpy(), *_transitions(t)[1:],
                                          precision=c["precision"])
            state["requests"].append((req, keep, c["types"], t["scan"]))
        state["in"] = None
        return state
    ctx = state["ctx"] = eels.Context(0)
    if kind in ("map", "request", "phonon"):
        ctx.set_association(case["grouping"])
        state["out"] = torch.empty((case["types"], case["nsy"], case["nsx"]), dtype=torch.float64,
                                   device="cuda")
    if kind == "phonon":
        state["configs"] = [_Workload(case, t) for t in sets]
    if kind == "elastic":
        ctx.set_exit_plane(True)
        state["out"] = torch.empty((len(DETECTORS), case["nsy"], case["nsx"]),
                                   dtype=torch.float64, device="cuda")
    if kind in ("map", "elastic"):
        state["sm"] = ctx.build_smatrix(s["vproj"], *_optics(case, s))
    if kind == "build":
        n_in = eels.count_beams(case["n"], case["cell"], LAM, case["f"], ALPHA)
        nh = case["n"] // 2
        state["out"] = torch.empty((case["n_z"], n_in, nh, nh), dtype=torch.complex64,
                                   device="cuda")
    return state


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(*r) for r in state["requests"]]
        return [srv.wait(i)[0] for i in ids]
    ctx, s, out = state["ctx"], state["in"][0], state["out"]
    if kind == "map":
        return ctx.inelastic_map(state["sm"], *_transitions(s), precision=c["precision"], out=out)
    if kind == "request":
        sm = ctx.build_smatrix(s["vproj"], *_optics(c, s))
        ctx.inelastic_map(sm, *_transitions(s), precision=c["precision"], out=out)
        sm.free()
        return out
    if kind == "phonon":
        return ctx.phonon_map(state["configs"], precision=c["precision"], out=out)
    if kind == "elastic":
        return ctx.elastic_images(state["sm"], s["scan"], DETECTORS, out=out)
    sm = ctx.build_smatrix(s["vproj"], *_optics(c, s))
    for depth in range(c["n_z"]):
        sm.copy_depth(depth, out[depth])
    sm.free()
    return out


# --- what a pass cannot do without -------------------------------------------------------

def _beams(c, angle):
    m = int(math.ceil(angle * c["cell"] / (LAM * c["f"]))) + 1
    return [(p, q) for q in range(-m, m + 1) for p in range(-m, m + 1)
            if LAM * c["f"] * math.sqrt(p * p + q * q) / c["cell"] <= angle]


def _usable(c):
    """Both apertures inside the band limit, as the calls require."""
    return all(16 * c["f"] ** 2 * (p * p + q * q) < c["n"] ** 2
               for k in _configurations(c) for p, q in _beams(k, BETA))


def _s_in_bytes(c):
    return max(8.0 * k["n_z"] * len(_beams(k, ALPHA)) * (k["n"] // 2) ** 2
               for k in _configurations(c))


def _contraction(c):
    """(complex multiply-adds of the cheaper grouping, sites that some probe sees)."""
    n_in, n_out = len(_beams(c, ALPHA)), len(_beams(c, BETA))
    layers, _ = _layers(c, np.random.default_rng(0))
    nsx, nsy, x0, y0, sx, sy = _scan(c)
    rx, ry = x0 + np.arange(nsx) * sx, y0 + np.arange(nsy) * sy
    first = last = seen = 0.0
    for xy, fe in layers:
        nr = [_in_window(xy[fe][:, k][:, None], r, c).sum(1) for k, r in ((0, rx), (1, ry))]
        nr = (nr[0] * nr[1]).astype(np.float64)
        nr = nr[nr > 0]
        seen += len(nr)
        p2, t = c["w"] ** 2, c["types"]
        first += float((t * n_out * n_in * (p2 + nr)).sum())
        last += float((nr * p2 * (n_in + t * n_out)).sum())
    return min(first, last), seen


def _in_window(site, probe, c):
    """The minimum-image rule: site - probe in [-L/2f, L/2f)."""
    d = site - probe
    d = d - c["cell"] * np.floor(d / c["cell"] + 0.5)
    h = c["cell"] / (2 * c["f"])
    return (d >= -h) & (d < h)


def work(case):
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _configurations(case):
        kind, n, nh, n_z = c["kind"], c["n"], c["n"] // 2, c["n_z"]
        n_in, n_out = len(_beams(c, ALPHA)), len(_beams(c, BETA))
        # one slice step of one band-limited wave: two N-point transforms per row, two per
        # column of the band
        step = 15.0 * n * n * math.log2(n)
        if kind in ("build", "request", "phonon"):
            total["bytes"] += 4.0 * n_z * n * n
            total["flops"] += step * n_z * n_in
        if kind == "build":
            total["bytes"] += 8.0 * n_z * n_in * nh * nh
        if kind in ("map", "request", "phonon"):
            macs, seen = _contraction(c)
            total["bytes"] += 8.0 * c["types"] * c["nsx"] * c["nsy"]
            total["bytes"] += 8.0 * c["types"] * c["w"] ** 2 * (1 if c["shared"] else seen)
            if kind == "map":   # the kept S-matrix: transmissions, and S_in in the windows
                total["bytes"] += 8.0 * n_z * n * n
                total["bytes"] += 8.0 * n_in * min(n_z * nh * nh, seen * c["w"] ** 2)
            total["flops"] += 8.0 * macs + step * n_z * n_out
        if kind == "elastic":
            cut, probes = nh // c["f"], c["nsx"] * c["nsy"]
            total["bytes"] += 8.0 * n_in * nh * nh + 8.0 * len(DETECTORS) * probes
            total["flops"] += probes * cut * cut * (8.0 * n_in + 10.0 * math.log2(cut))
    return total


def _cost(c):
    """Rough seconds of a pass, to keep drawn cases within the listed ones."""
    rate = {"fp32": 1.0e13, "tf32": 2.5e14, "bf16x3": 5.0e14, "": 1.0e13}[c["precision"]]
    total = 0.0
    for k in _configurations(c):
        n_in, n_out = len(_beams(k, ALPHA)), len(_beams(k, BETA))
        step = 15.0 * k["n"] ** 2 * math.log2(k["n"]) / 2.0e13
        if k["kind"] in ("build", "request", "phonon"):
            total += step * k["n_z"] * n_in
        if k["kind"] in ("map", "request", "phonon"):
            total += 8.0 * _contraction(k)[0] / rate + step * k["n_z"] * n_out
        if k["kind"] == "elastic":
            total += 8.0 * k["nsx"] * k["nsy"] * (k["n"] // 2 // k["f"]) ** 2 * n_in / rate
    return total


# --- the same results in 64 bits ---------------------------------------------------------

def exact(case, seed):
    if _seconds64(case) > 12.0:
        return None
    rng = np.random.default_rng(seed)
    sets = [(c, _inputs(c, rng)) for c in _configurations(case)]
    kind = case["kind"]
    with torch.no_grad():
        if kind == "build":
            return _s_in64(*sets[0])[0]
        if kind == "elastic":
            return _images64(*sets[0])
        maps = [_map64(c, s) for c, s in sets]
    if kind == "serve":
        return maps
    return sum(maps) / len(maps)


def _seconds64(case):
    """Rough time of exact() at 0.8 FP64 TFLOP/s."""
    total = 0.0
    for c in _configurations(case):
        waves = len(_beams(c, ALPHA)) + (len(_beams(c, BETA)) if c["w"] else 0)
        total += 25.0 * c["n"] ** 2 * math.log2(c["n"]) * c["n_z"] * waves
        if c["w"]:
            total += 8.0 * _contraction(c)[0]
        if c["kind"] == "elastic":
            total += 8.0 * c["nsx"] * c["nsy"] * (c["n"] // 2) ** 2 * len(_beams(c, ALPHA))
    return total / 0.8e12


def _tables64(c, s):
    n = c["n"]
    t = torch.exp(1j * SIGMA * s["vproj"].double())
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    k2 = k[:, None] ** 2 + k[None, :] ** 2
    phase = torch.remainder(LAM * s["dz"] * k2 / c["cell"] ** 2, 2.0)
    return t, torch.exp(-1j * math.pi * phase) * (16 * k2 < n * n)


def _plane64(c, beams):
    """Unit-norm plane waves of the beams, [beam][n][n]."""
    n, f = c["n"], c["f"]
    psi = torch.zeros((len(beams), n, n), dtype=torch.complex128, device="cuda")
    for j, (p, q) in enumerate(beams):
        psi[j, (f * q) % n, (f * p) % n] = 1.0
    return torch.fft.ifft2(psi, norm="ortho")


def _groups(c, beams):
    """Beams in groups of about 4 GB of waves."""
    m = max(1, int(4e9 / (16 * c["n"] ** 2)))
    return [beams[i:i + m] for i in range(0, len(beams), m)]


def _s_in64(c, s):
    """S_in at every depth in the library's scale (N times the decimated wave t psi), and the
    decimated exit waves."""
    t, prop = _tables64(c, s)
    parts, ends = [], []
    for beams in _groups(c, _beams(c, ALPHA)):
        psi, depth = _plane64(c, beams), []
        for i in range(c["n_z"]):
            psi = psi * t[i]
            depth.append(c["n"] * psi[:, ::2, ::2])
            psi = torch.fft.ifft2(torch.fft.fft2(psi) * prop)
        parts.append(torch.stack(depth))
        ends.append(psi[:, ::2, ::2].clone())
    return torch.cat(parts, 1), torch.cat(ends)


def _coefficients64(c, rx, ry):
    b = torch.tensor(_beams(c, ALPHA), device="cuda", dtype=torch.float64)
    ph = [torch.exp(-2j * math.pi * c["f"] / c["cell"] * b[:, k][:, None]
                    * torch.from_numpy(r).cuda()[None, :]) for k, r in ((0, rx), (1, ry))]
    return ph[0] * (c["f"] / math.sqrt(len(b))), ph[1]


def _map64(c, s):
    """I(R) = f^2 sum over sites and detector beams |sum_p conj(S_out) H S_in a(R)|^2."""
    n, nh, w, f = c["n"], c["n"] // 2, c["w"], c["f"]
    t, prop = _tables64(c, s)
    s_in, _ = _s_in64(c, s)
    nsx, nsy, x0, y0, sx, sy = s["scan"]
    rx, ry = x0 + np.arange(nsx) * sx, y0 + np.arange(nsy) * sy
    ax, ay = _coefficients64(c, rx, ry)
    out = torch.zeros((c["types"], nsy, nsx), dtype=torch.float64, device="cuda")
    u = torch.arange(w, device="cuda")
    for beams in _groups(c, _beams(c, BETA)):
        beta = torch.fft.ifft2(torch.fft.fft2(_plane64(c, beams)) * prop.conj())
        for i in range(c["n_z"] - 1, -1, -1):
            s_out = 4.0 * beta[:, ::2, ::2]
            for k in np.nonzero(s["slice"] == i)[0]:
                okx = np.nonzero(_in_window(s["x"][k], rx, c))[0]
                oky = np.nonzero(_in_window(s["y"][k], ry, c))[0]
                if not len(okx) or not len(oky):
                    continue
                rows, cols = (int(s["wy"][k]) + u) % nh, (int(s["wx"][k]) + u) % nh
                b = s_out[:, rows][:, :, cols].reshape(len(beams), -1).conj()
                a = s_in[i][:, rows][:, :, cols].reshape(s_in.shape[1], -1) / n
                ix, iy = torch.from_numpy(okx).cuda(), torch.from_numpy(oky).cuda()
                coef = (ay[:, iy][:, :, None] * ax[:, ix][:, None, :]).reshape(len(a), -1)
                many = coef.shape[1] > a.shape[1]
                probe = None if many else a.t() @ coef
                for m in range(c["types"]):
                    h = (s["H"][m] if c["shared"] else s["H"][k, m]).to(torch.complex128)
                    hb = b * h.reshape(-1)
                    v = (hb @ a.t()) @ coef if many else hb @ probe
                    got = f * f * (v.real ** 2 + v.imag ** 2).sum(0).reshape(len(iy), len(ix))
                    out[m].index_put_((iy[:, None], ix[None, :]), got, accumulate=True)
            if i:
                beta = torch.fft.ifft2(torch.fft.fft2(beta * t[i].conj()) * prop.conj())
    return out


def _images64(c, s):
    """f^2-normalised diffraction intensity of each probe's L/f cut inside the detectors."""
    n, nh, f = c["n"], c["n"] // 2, c["f"]
    cut = nh // f
    _, ends = _s_in64(c, s)
    nsx, nsy, x0, y0, sx, sy = s["scan"]
    rx, ry = x0 + np.arange(nsx) * sx, y0 + np.arange(nsy) * sy
    ax, ay = _coefficients64(c, rx, ry)

    def pixels(r):
        ok = _in_window(np.arange(nh) * (c["cell"] / nh), r, c)
        first = 0 if ok.all() else int(np.nonzero(ok & ~np.roll(ok, 1))[0][0])
        return (first + torch.arange(cut, device="cuda")) % nh

    k = torch.fft.fftfreq(cut, 1.0 / cut, device="cuda", dtype=torch.float64)
    k2 = k[:, None] ** 2 + k[None, :] ** 2
    angle = LAM * f * torch.sqrt(k2) / c["cell"]
    band = 16 * f * f * k2 < n * n
    masks = [band & (angle >= lo) & ((angle <= hi) if hi > 0 else band) for lo, hi in DETECTORS]
    out = torch.zeros((len(masks), nsy, nsx), dtype=torch.float64, device="cuda")
    for iy in range(nsy):
        rows = ends[:, pixels(ry[iy])] * ay[:, iy][:, None, None]
        exit_waves = (ax.t() @ rows.reshape(len(rows), -1)).reshape(nsx, cut, nh)
        for ix in range(nsx):
            spec = torch.fft.fft2(exit_waves[ix][:, pixels(rx[ix])])
            p = spec.real ** 2 + spec.imag ** 2
            for d, mask in enumerate(masks):
                out[d, iy, ix] = 16.0 * f * f / (n * n) * p[mask].sum()
    return out
