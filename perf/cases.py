"""The work users have this library do, as timed cases.

Every case goes through the package's public entry points (``StressContext``,
``StressGraph``): single evaluations from the smallest disk to the full polycrystalline
layer, ragged and tall grids, batches with reduced storage, captured sweeps, the
server's family subsets, host buffers, the per-height statistics, the free-surface
relaxation, and new geometries (interaction coefficients and their spectra built, then
used).  Sizes, cells and families are those of ``workloads`` and of the tests.

``exact`` evaluates the same quantities in 64 bits with plain torch: the coefficients
from Eq. 6 / 9b with the near cells subdivided, the convolution by a padded FFT, the
relaxation by its difference equations.
"""
import math

import numpy as np
import torch

import paper_1804_01830_gb300 as dds

UM = 1.0e-6
MU, NU = 68.0e9, 0.23
A, C = 0.319e-9, 0.519e-9          # a- and c-type Burgers lengths
CM2 = 1.0e4

# ------------------------------------------------------------------ families ---


def _hex(i):
    return [A * math.cos(math.radians(60.0 * i)), A * math.sin(math.radians(60.0 * i)), 0.0]


def families(kind):
    """(t, b) of a family set: "edge" one vertical edge family; "disk" the edge and the
    mixed family of the radial disk; "gan" the 18 families of the GaN-like layer;
    "hexedge" its six vertical edge families; "mixed" three families of two line
    directions without a common mirror plane; "five" five families of two directions."""
    z = [0.0, 0.0, 1.0]
    s, c = math.sin(math.radians(15.6)), math.cos(math.radians(15.6))
    t = [z] * 6 + [[0.0, s, c]] * 12
    b = [_hex(i) for i in range(6)]
    for i in range(6):
        for sign in (1.0, -1.0):
            b.append([_hex(i)[0], _hex(i)[1], sign * C])
    pick = {"gan": range(18), "hexedge": range(6), "mixed": (0, 7, 8), "five": (1, 4, 6, 13, 17)}
    if kind in pick:
        return np.array([t[f] for f in pick[kind]]), np.array([b[f] for f in pick[kind]])
    r3 = math.sqrt(3.0)
    t2, b2 = [[0.0, 0.0, 1.0], [0.0, 0.5, r3 / 2.0]], [[A, 0.0, 0.0], [A / 2.0, r3 * A / 2.0, C]]
    n = {"edge": 1, "disk": 2}[kind]
    return np.array(t2[:n]), np.array(b2[:n])


def n_fields(kind):
    """Distinct Cartesian density fields a family set needs (the coefficients are linear in b)."""
    return {"edge": 1, "disk": 2, "gan": 5, "hexedge": 2, "mixed": 3, "five": 5}[kind]


# --------------------------------------------------------------------- cases ---
def _case(name, call, grid, cells, fam, **more):
    d = {"name": name, "call": call, "nx": grid[0], "ny": grid[1], "nz": grid[2], "dx": cells[0] * UM,
         "dy": cells[1] * UM, "dz": cells[2] * UM, "families": fam, "density": "grains", "dtype": "f32",
         "fp16_spectra": False, "shells": 0, "periodic": False, "sets": 1, "steps": 0, "present": 0}
    d.update(more)
    return d


GAN = (0.2, 0.2, 0.05)


def listed():
    return [
        # one dislocation type in a small disk: the smallest call, latency and launches
        _case("disk_32x32x8", "stress", (32, 32, 8), (1.0, 1.0, 0.25), "edge", density="disk"),
        # the radially varying disk: a thin wide grid, two families
        _case("radial_disk_512x512x16", "stress", (512, 512, 16), (0.5, 0.5, 0.2), "disk", density="disk"),
        # the polycrystalline GaN-like layer with its 18 families: the headline evaluation
        _case("gan_layer_256x256x128", "stress", (256, 256, 128), GAN, "gan"),
        # a tall column of ragged sizes with families of no common mirror plane
        _case("tall_90x77x200", "stress", (90, 77, 200), (0.2, 0.2, 0.1), "mixed"),
        # a thin polycrystalline film of odd sizes with its per-height statistics (Eq. 20)
        _case("film_stats_250x241x29", "stats", (250, 241, 29), GAN, "gan"),
        # four grain realisations on one context, both reduced storage options
        _case("batch_128x128x128x4", "multi", (128, 128, 128), GAN, "gan", sets=4, dtype="bf16", fp16_spectra=True),
        # grain-size sweep: realisations on two grids replayed as one captured graph
        _case("sweep_graph_128_256x64", "graph", (128, 128, 64), GAN, "gan", sets=3),
        # two requests of the server on its largest grid, three of the 18 families present
        _case("serving_512x512x64x2", "subset", (512, 512, 64), (0.2, 0.2, 0.05), "gan", sets=2, present=3),
        # densities and stresses in (pinned) host memory, copies included
        _case("host_128x128x128", "host", (128, 128, 128), GAN, "gan"),
        # relaxation of the layer to free surfaces (Sec. 5), total stress at the end
        _case("relax_256x256x128", "relax", (256, 256, 128), GAN, "gan", steps=20),
        # a geometry the server has not seen (or has evicted): coefficients, spectra, first stress
        _case("new_geometry_128x128x64", "build", (128, 128, 64), GAN, "gan"),
        # one point of the grain-size study (Sec. 6.4): replica sums of 15 shells, then its fluctuations
        _case("grain_study_64x64x8", "build", (64, 64, 8), (0.625, 0.625, 0.25), "hexedge", shells=15),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["stress", "stress", "stress", "stats", "multi", "graph", "subset", "host", "relax", "build"])
    while True:
        nx, ny, nz = _log_int(rng, 8, 512), _log_int(rng, 8, 512), _log_int(rng, 2, 256)
        if rng.random() < 0.3:                          # the powers of two that layers are often given
            nx, ny, nz = (1 << round(math.log2(v)) for v in (nx, ny, nz))
        pad = 1
        for n in (nx, ny, nz):
            pad *= 1 << math.ceil(math.log2(2 * n))
        if 4096 <= pad <= 1 << 25:
            break
    dx = rng.choice([0.2, 0.5, 1.0])
    case = _case("", call, (nx, ny, nz), (dx, dx, dx * rng.choice([0.1, 0.25, 0.5, 1.0])),
                 rng.choice(["edge", "disk", "gan", "gan", "gan", "hexedge", "mixed", "five"]))
    del case["name"]
    case["density"] = rng.choice(["disk", "grains"])
    if call in ("stress", "stats", "multi", "graph", "subset"):
        case["dtype"] = rng.choice(["f32", "f32", "f32", "bf16"])
    if call in ("stress", "multi"):
        case["fp16_spectra"] = rng.random() < 0.2
    if call in ("multi", "graph", "subset", "stats"):
        case["sets"] = rng.randint(1, max(1, min(4, (1 << 25) // pad)))
    if call == "subset":
        case["present"] = rng.randint(1, min(4, len(families(case["families"])[0])))
    if call == "relax":
        case["steps"] = rng.randint(5, 25)
    if call in ("stress", "stats", "build") and pad <= 1 << 20 and rng.random() < 0.3:
        case["shells"] = rng.randint(1, 3)
        if ny >= 32 and ny & (ny - 1) == 0:
            case["periodic"] = rng.random() < 0.5
    return case


# -------------------------------------------------------------------- inputs ---
def _parts(case):
    """Grids evaluated by one pass, as (nx, ny, nz, density sets)."""
    g = (case["nx"], case["ny"], case["nz"], case["sets"])
    if case["call"] == "graph":                         # a second grid of twice the width, one set
        return [g, (min(512, 2 * case["nx"]), min(512, 2 * case["ny"]), case["nz"], 1)]
    return [g]


def _n_input_families(case):
    return case["present"] or len(families(case["families"])[0])


def _present(case):
    """The families with density, spread over the context's families."""
    F = len(families(case["families"])[0])
    n = _n_input_families(case)
    return [(i * F) // n for i in range(n)]


def _density(case, seed, part, device="cuda"):
    """(sets, F, nz, ny, nx) line densities in 1/m^2: grains carry the GaN layer's height
    profile, each at its own level, in one or two of the families; the disk is the radial
    profile, scaled per family."""
    nx, ny, nz, sets = _parts(case)[part]
    F = _n_input_families(case)
    gen = torch.Generator().manual_seed(1000003 * int(seed) + part)
    x = (torch.arange(nx, dtype=torch.float32) + 0.5).to(device)
    y = (torch.arange(ny, dtype=torch.float32) + 0.5).to(device)
    z = ((torch.arange(nz, dtype=torch.float32) + 0.5) * (case["dz"] / (0.5 * UM))).to(device)
    out = torch.empty((sets, F, nz, ny, nx), dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32,
                      device=device)
    for s in range(sets):
        u = torch.rand(1 + F, generator=gen).tolist()
        if case["density"] == "disk":
            r2 = ((x - 0.5 * nx) / (0.47 * nx)) ** 2 + ((y[:, None] - 0.5 * ny) / (0.47 * ny)) ** 2
            plane = torch.where(r2 < 1.0, 1.0 + (2.0 + 4.0 * u[0]) * r2, torch.zeros_like(r2))
            for f in range(F):
                out[s, f] = (1.0e9 * CM2 * (0.5 + u[1 + f])) * plane
            continue
        prof = (1.0e10 * torch.exp(-z) + 1.0e8) * CM2
        area = nx * case["dx"] * ny * case["dy"]
        grain = (0.5 + 3.0 * u[0]) * UM if case["shells"] == 0 else 0.1 * nx * case["dx"]
        k = max(1, min(2048, int(round(area / (math.pi / 4.0 * grain * grain)))))
        sx = (torch.rand(k, generator=gen) * nx).to(device)
        sy = (torch.rand(k, generator=gen) * ny).to(device)
        owner = torch.empty((ny, nx), dtype=torch.int64, device=device)
        for j in range(0, ny, 32):                      # nearest seed of every column
            d = (x[None, :, None] - sx) ** 2 + (y[j:j + 32, None, None] - sy) ** 2
            owner[j:j + 32] = d.argmin(dim=2)
        prof = prof[:, None, None] * (0.5 + torch.rand(k, generator=gen)).to(device)[owner]
        one = torch.randint(0, F, (k,), generator=gen).to(device)[owner]
        two = torch.randint(0, F, (k,), generator=gen).to(device)[owner]
        for f in range(F):
            out[s, f] = prof * ((one == f) | (two == f)).to(torch.float32)
    return out


def _load(case, seed, device="cuda"):
    """Stress of the dislocations for the relaxation: a few smooth modes, 100 MPa."""
    nx, ny, nz, _ = _parts(case)[0]
    gen = torch.Generator().manual_seed(1000003 * int(seed) + 17)
    x = (torch.arange(nx, dtype=torch.float64) * (2.0 * math.pi / nx)).to(device)
    y = (torch.arange(ny, dtype=torch.float64) * (2.0 * math.pi / ny)).to(device)[:, None]
    z = (torch.arange(nz, dtype=torch.float64) * (math.pi / nz)).to(device)[:, None, None]
    out = torch.empty((6, nz, ny, nx), dtype=torch.float32, device=device)
    for c in range(6):
        f = torch.zeros((nz, ny, nx), dtype=torch.float64, device=device)
        for _ in range(3):
            k = torch.randint(1, 5, (3,), generator=gen).tolist()
            p = (2.0 * math.pi * torch.rand(3, generator=gen)).tolist()
            f += torch.sin(k[0] * x + p[0]) * torch.cos(k[1] * y + p[1]) * torch.cos(k[2] * z + p[2])
        out[c] = (1.0e8 * f).to(torch.float32)
    return out


def _context(case, part=0):
    nx, ny, nz, _ = _parts(case)[part]
    ctx = dds.StressContext(0)
    ctx.set_geometry(nx, ny, nz, case["dx"], case["dy"], case["dz"], MU, NU)
    ctx.set_families(*families(case["families"]))
    if case["fp16_spectra"]:
        ctx.set_option(dds.DDS_OPT_SPECTRA_FP16, 1)
    if case["shells"]:
        ctx.set_option(dds.DDS_OPT_PBC_SHELLS, case["shells"])
        ctx.set_option(dds.DDS_OPT_PBC_PERIODIC, int(case["periodic"]))
    return ctx


def prepare(case, seed):
    call = case["call"]
    st = {"case": case}
    if call == "relax":
        st["ctx"] = _context(case)
        st["sigma_dis"] = _load(case, seed)
        return st
    rho = [_density(case, seed, p) for p in range(len(_parts(case)))]
    if call == "build":
        st["rho"] = rho[0][0].contiguous()
        st["ctx"] = None
        return st
    st["ctx"] = [_context(case, p).build_kernels() for p in range(len(rho))]
    if call == "graph":
        st["graph"] = dds.StressGraph(list(zip(st["ctx"], rho)))
    elif call == "host":
        st["rho"] = rho[0][0].to("cpu").pin_memory().numpy()
        st["sigma"] = torch.empty((6,) + tuple(rho[0].shape[2:]), dtype=torch.float32).pin_memory().numpy()
    elif call == "stress":
        st["rho"] = rho[0][0].contiguous()
        st["sigma"] = torch.empty((6,) + tuple(rho[0].shape[2:]), dtype=torch.float32, device="cuda")
    else:
        st["rho"] = rho[0]
        st["sigma"] = torch.empty((rho[0].shape[0], 6) + tuple(rho[0].shape[2:]), dtype=torch.float32, device="cuda")
    return st


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "relax":
        return list(state["ctx"].relax(state["sigma_dis"], case["steps"]))
    if call == "build":
        if state["ctx"] is not None:                    # the geometry that makes room
            state["ctx"].close()
        state["ctx"] = _context(case).build_kernels()
        return list(state["ctx"].stress_stats(state["rho"]))
    ctx = state["ctx"][0]
    if call == "stress":
        return ctx.stress(state["rho"], state["sigma"])
    if call == "multi":
        return ctx.stress_multi(state["rho"], state["sigma"])
    if call == "subset":
        return ctx.stress_subset(_present(case), state["rho"], state["sigma"])
    if call == "stats":
        return list(ctx.stress_stats(state["rho"], state["sigma"]))
    if call == "graph":
        state["graph"].launch()
        return list(state["graph"].sigma)
    return ctx.stress_host(state["rho"], state["sigma"])


def work(case):
    """Densities read and stresses written once (the interaction is not counted: it could
    be held in many forms); the operations of the real FFTs on the doubled grid and of
    the product in Fourier space; for a build, those of one field evaluation per offset
    and replica and of the transforms; per relaxation step, u and its force read, u written."""
    nbytes = flops = 0.0
    fe = n_fields(case["families"])
    for nx, ny, nz, sets in _parts(case):
        cells = float(nx * ny * nz)
        if case["call"] == "relax":
            nbytes += cells * (24 + 24 + 24 + 36.0 * case["steps"])
            flops += cells * 100.0 * case["steps"]
            continue
        pad = 8.0 * cells
        fft = 2.5 * pad * math.log2(pad)
        el = 2 if case["dtype"] == "bf16" else 4
        nbytes += sets * cells * (el * _n_input_families(case) + 24)
        flops += sets * (fft * (fe + 6) + 4.0 * 6 * fe * pad / 2)
        if case["call"] == "build":
            images = (2.0 * case["shells"] + 1) ** 2
            flops += pad / 2 * images * (150.0 + 100.0 * fe) + 6 * fe * fft / 2
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------- 64-bit values, torch ---
PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))     # xx yy zz xy xz yz


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _segment_end(R, t, b):
    """Bracket of Eq. 6 at one end of the segment."""
    Rn = torch.sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2])
    L = R[0] * t[0] + R[1] * t[1] + R[2] * t[2]
    Rt = [R[a] + Rn * t[a] for a in range(3)]
    inv = 1.0 / (Rt[0] * Rt[0] + Rt[1] * Rt[1] + Rt[2] * Rt[2])
    perp = [R[a] - L * t[a] for a in range(3)]
    u, w = _cross(b, Rt), _cross(b, t)
    k1 = 1.0 / (1.0 - NU)
    k2 = 0.5 * k1 * (u[0] * t[0] + u[1] * t[1] + u[2] * t[2])
    ratio = L / Rn
    out = []
    for a, c in PAIRS:
        s1 = 0.5 * (u[a] * t[c] + u[c] * t[a])
        s2 = 0.5 * (w[a] * Rt[c] + w[c] * Rt[a])
        phi = 2.0 * inv * (perp[a] * Rt[c] + perp[c] * Rt[a] + ratio * Rt[a] * Rt[c])
        out.append(inv * (s1 - k1 * s2 - k2 * ((1.0 if a == c else 0.0) + t[a] * t[c] + phi)))
    return out


def _box(r, h, t, b):
    """Coefficient of a box of edges h at observer offset r (Eq. 9b times its volume)."""
    dl = min(h[a] / abs(t[a]) for a in range(3) if t[a] != 0.0)
    ends = [[-0.5 * dl * t[a] - r[a] for a in range(3)], [0.5 * dl * t[a] - r[a] for a in range(3)]]
    cosines = [sum(E[a] * t[a] for a in range(3)) / torch.sqrt(sum(E[a] * E[a] for a in range(3))) for E in ends]
    flip = torch.where(cosines[0] + cosines[1] < 0.0, -1.0, 1.0).to(torch.float64)
    SA, SB = ([s for s in _segment_end([flip * E[a] for a in range(3)], t, b)] for E in ends)
    f = MU / math.pi * h[0] * h[1] * h[2] / dl
    zero = (r[0] == 0.0) & (r[1] == 0.0) & (r[2] == 0.0)
    return torch.stack([torch.where(zero, torch.zeros_like(p), f * (p - q)) for p, q in zip(SB, SA)])


def _subcells(h):
    out = []
    for a in range(3):
        r = h[a] / min(h)
        lo = max(1, int(math.floor(r)))
        out.append(lo + 1 if lo * (lo + 1) <= r * r else lo)
    return out


def _cells(i, j, k, h, t, b):
    """Coefficients (6, n) at cell offsets (flat integer tensors); near cells subdivided."""
    d = [i.double() * h[0], j.double() * h[1], k.double() * h[2]]
    out = _box(d, h, t, b)
    near = torch.nonzero(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] < (3.0 * max(h)) ** 2).flatten()
    if near.numel():
        m = _subcells(h)
        hs = [h[a] / m[a] for a in range(3)]
        q = [torch.arange(1 - m[a], m[a], device=i.device) for a in range(3)]
        gx, gy, gz = torch.meshgrid(*q, indexing="ij")
        mult = ((m[0] - gx.abs()) * (m[1] - gy.abs()) * (m[2] - gz.abs())).double().flatten()
        sub = [gx.flatten().double() * hs[0], gy.flatten().double() * hs[1], gz.flatten().double() * hs[2]]
        step = max(1, (1 << 22) // mult.numel())
        for s in range(0, near.numel(), step):
            at = near[s:s + step]
            r = [d[a][at][:, None] + sub[a][None, :] for a in range(3)]
            out[:, at] = (_box(r, hs, t, b) * mult).sum(dim=2) / (m[0] * m[1] * m[2])
    return out


def _images(i, n):
    """Minimal image of an offset for period n: pairs (offset, weight), ties averaged."""
    m = torch.remainder(i, n)
    r = torch.where(2 * m > n, m - n, m)
    tie = 2 * m == n
    if not bool(tie.any()):
        return [(r, torch.ones_like(r, dtype=torch.float64))]
    w = torch.where(tie, 0.5, 1.0).double()
    return [(r, w), (-r, torch.where(tie, 0.5, 0.0).double())]


def _table(case, grid, t, b):
    """Coefficients at every offset, wrapped into the doubled grid: (6, 2 nz, 2 ny, 2 nx)."""
    nx, ny, nz = grid
    h = [case["dx"], case["dy"], case["dz"]]
    dev = "cuda"

    def wrapped(n):
        q = torch.arange(2 * n, device=dev)
        return torch.where(q < n, q, q - 2 * n), q != n

    (ix, okx), (iy, oky), (iz, okz) = wrapped(nx), wrapped(ny), wrapped(nz)
    out = torch.empty((6, 2 * nz, 2 * ny, 2 * nx), dtype=torch.float64, device=dev)
    n = case["shells"]
    rows = max(1, (1 << 22) // (4 * nx * ny))
    for s in range(0, 2 * nz, rows):
        kk, jj, ii = torch.meshgrid(iz[s:s + rows], iy, ix, indexing="ij")
        ok = (okz[s:s + rows, None, None] & oky[:, None] & okx).flatten()
        shape = kk.shape
        i, j, k = ii.flatten(), jj.flatten(), kk.flatten()
        if n == 0:
            v = _cells(i, j, k, h, t, b)
        else:
            xs = _images(i, nx) if case["periodic"] else [(i, None)]
            ys = _images(j, ny) if case["periodic"] else [(j, None)]
            v = torch.zeros((6, i.numel()), dtype=torch.float64, device=dev)
            for xi, wx in xs:
                for yj, wy in ys:
                    w = 1.0 if wx is None else wx * wy
                    for p in range(-n, n + 1):
                        for q in range(-n, n + 1):
                            v += w * _cells(xi + p * nx, yj + q * ny, k, h, t, b)
        out[:, s:s + rows] = torch.where(ok, v, torch.zeros_like(v)).reshape((6,) + shape)
    return out


def _exact_stress(case, seed, part):
    """sigma (sets, 6, nz, ny, nx) in 64 bits."""
    nx, ny, nz, sets = _parts(case)[part]
    t, b = families(case["families"])
    if case["call"] == "subset":
        t, b = t[_present(case)], b[_present(case)]
    rho = _density(case, seed, part)
    shape = (2 * nz, 2 * ny, 2 * nx)
    acc = torch.zeros((sets, 6, 2 * nz, 2 * ny, nx + 1), dtype=torch.complex128, device="cuda")
    directions = {tuple(v) for v in t.tolist()}
    for d in sorted(directions):
        members = [f for f in range(len(t)) if tuple(t[f]) == d]
        for a in range(3):
            if all(b[f][a] == 0.0 for f in members):
                continue
            unit = [A if c == a else 0.0 for c in range(3)]
            table = _table(case, (nx, ny, nz), list(d), unit)
            fields = torch.zeros((sets, nz, ny, nx), dtype=torch.float64, device="cuda")
            for f in members:
                fields += (b[f][a] / A) * rho[:, f].double()
            hats = [torch.fft.rfftn(fields[s], s=shape) for s in range(sets)]
            for c in range(6):
                g = torch.fft.rfftn(table[c])
                for s in range(sets):
                    acc[s, c] += g * hats[s]
            del table, fields, hats, g
    del rho
    out = torch.empty((sets, 6, nz, ny, nx), dtype=torch.float64, device="cuda")
    for s in range(sets):
        for c in range(6):
            out[s, c] = torch.fft.irfftn(acc[s, c], s=shape)[:nz, :ny, :nx]
    return out


def _exact_relax(case, seed):
    """(u, sigma_tot) of the explicit relaxation (Eqs. 14-18) in 64 bits."""
    h = [case["dx"], case["dy"], case["dz"]]
    E = 2.0 * MU * (1.0 + NU)
    lam2 = E * (1.0 - NU) / ((1.0 + NU) * (1.0 - 2.0 * NU))
    shear = E / (2.0 * (1.0 + NU))
    dt = min(h) ** 2 / (5.0 * lam2 - 3.0 * shear)
    sig = _load(case, seed).double()
    nz = sig.shape[1]
    index = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}

    def s(a, c):
        return sig[index[(min(a, c), max(a, c))]]

    def central(f, axis):                               # periodic in x and y; arrays [..., z, y, x]
        dim = -1 - axis
        return (torch.roll(f, -1, dim) - torch.roll(f, 1, dim)) / (2.0 * h[axis])

    def dz_onesided(f):
        if nz < 3:
            return ((f[1] - f[0]) / h[2]).expand_as(f)
        d = torch.empty_like(f)
        d[1:-1] = (f[2:] - f[:-2]) / (2.0 * h[2])
        d[0] = (-3.0 * f[0] + 4.0 * f[1] - f[2]) / (2.0 * h[2])
        d[-1] = (3.0 * f[-1] - 4.0 * f[-2] + f[-3]) / (2.0 * h[2])
        return d

    force = torch.stack([central(s(a, 0), 0) + central(s(a, 1), 1) + dz_onesided(s(a, 2)) for a in range(3)])
    ps, pn = -(1.0 + NU) / E, -(1.0 + NU) * (1.0 - 2.0 * NU) / E

    def ghosts(u):
        """u with one layer below and above the film (Eq. 18b)."""
        e = torch.empty((3, nz + 2) + tuple(u.shape[2:]), dtype=torch.float64, device=u.device)
        e[:, 1:-1] = u
        for layer, inner, row, sign in ((0, 1, 0, -1.0), (nz - 1, nz - 2, nz + 1, 1.0)):
            e[0, row] = u[0, inner] + sign * 2.0 * h[2] * (2.0 * ps * s(0, 2)[layer] - central(u[2, layer], 0))
            e[1, row] = u[1, inner] + sign * 2.0 * h[2] * (2.0 * ps * s(1, 2)[layer] - central(u[2, layer], 1))
            e[2, row] = u[2, inner] + sign * 2.0 * h[2] / (1.0 - NU) * (
                pn * s(2, 2)[layer] - NU * (central(u[0, layer], 0) + central(u[1, layer], 1)))
        return e

    def second(e, axis):
        if axis == 2:
            return (e[2:] - 2.0 * e[1:-1] + e[:-2]) / h[2] ** 2
        f = e[1:-1]
        return (torch.roll(f, -1, -1 - axis) - 2.0 * f + torch.roll(f, 1, -1 - axis)) / h[axis] ** 2

    def mixed(e, a, c):
        if 2 not in (a, c):
            return central(central(e[1:-1], a), c)
        return central((e[2:] - e[:-2]) / (2.0 * h[2]), a if c == 2 else c)

    u = torch.zeros((3,) + tuple(sig.shape[1:]), dtype=torch.float64, device=sig.device)
    for _ in range(case["steps"]):
        e = ghosts(u)
        new = torch.empty_like(u)
        for a in range(3):
            r = force[a].clone()
            for c in range(3):
                r += (lam2 if a == c else shear) * second(e[a], c)
                if c != a:
                    r += (lam2 - shear) * mixed(e[c], a, c)
            new[a] = u[a] + dt * r
        u = new
    e = ghosts(u)
    grad = [[central(u[a], 0), central(u[a], 1), (e[a, 2:] - e[a, :-2]) / (2.0 * h[2])] for a in range(3)]
    div = (lam2 - 2.0 * shear) * (grad[0][0] + grad[1][1] + grad[2][2])
    tot = sig.clone()
    for q, (a, c) in enumerate(PAIRS):
        tot[q] += shear * (grad[a][c] + grad[c][a])
        if a == c:
            tot[q] += div
    return u, tot


def exact(case, seed):
    call = case["call"]
    if call == "relax":
        return list(_exact_relax(case, seed))
    sig = [_exact_stress(case, seed, p) for p in range(len(_parts(case)))]
    if call == "graph":
        return sig
    if call in ("stress", "host"):
        return sig[0][0].cpu().numpy() if call == "host" else sig[0][0]
    if call in ("stats", "build"):
        s = torch.sqrt((sig[0] ** 2).mean(dim=(3, 4)))
        return [sig[0], s] if call == "stats" else [sig[0][0], s[0]]
    return sig[0]
