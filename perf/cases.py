"""The cases that this framework's speed is measured on: MSM evaluations, their
gradients, replica batches and molecular dynamics, each through the calls that
a program makes, over the sizes that the repository's workloads span (a few
thousand atoms to 4.1 million).

A case names a system (kind of box, atoms, box edges), the MSM parameters, the
precision of the plan and what is asked of it.  Inputs are water boxes at
0.1 atoms per cubic Angstrom with a few ions (rigid TIP3P geometry on a
jittered lattice), or a plasma of like charges for molecular dynamics, drawn on
the GPU from the seed.

A program on a mixed plan holds its positions, charges and results in single
precision (the plan computes pairs and grids in FP32, so its results carry no
more), its energy, one FP64 number, joining the others.  The batch graph
writes FP64 buffers; the program keeps its samples in single precision too.  A
program on an FP64 plan holds everything in FP64.

``exact`` is the same method (the same splitting, grids and basis functions)
written in plain torch in 64 bits.
"""
import math

import torch

from paper_1402_7216_gb300 import MSM, MSMBatch, MSMEnergy

DEV = "cuda" if torch.cuda.is_available() else "cpu"
DENSITY = 0.1  # atoms per cubic Angstrom
SPACING_OF_SITES = 2.5  # Angstrom, the least distance of two oxygens or ions

# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------


def _case(name, what, atoms, box, precision="mixed", periodic=True, cutoff=10.0, spacing=2.0, levels=0, order=3,
          splitting=2, ions=0, **more):
    lx, ly, lz = box if isinstance(box, tuple) else (box,) * 3
    c = dict(what=what, atoms=atoms, lx=lx, ly=ly, lz=lz, precision=precision, periodic=periodic, cutoff=cutoff,
             spacing=spacing, levels=levels, order=order, splitting=splitting, ions=ions, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest real system, a water droplet in an open box: energies and
        # forces of a step of a small simulation, where launches and latency count
        _case("forces_open_3k", "forces", 3000, 30.0, periodic=False, cutoff=12.0, spacing=2.5, splitting=1),
        # the common solvated-protein size, forces for a simulation step
        _case("forces_23k", "forces", 23558, 62.2, ions=2),
        # the same box in training: energy as a loss, gradients with respect to
        # positions and charges through autograd
        _case("gradients_23k", "gradients", 23558, 62.2, ions=2),
        # a mid-sized box with three different edges and an odd atom count,
        # quintic basis, C3 smoothing
        _case("forces_191k_ragged", "forces", 190977, (131.3, 118.9, 122.4), spacing=1.8, order=5, splitting=3,
              ions=330),
        # the benchmark system: 216.8 A box, 0.15 M salt, quintic
        _case("forces_1m", "forces", 1066628, 216.8, cutoff=12.0, spacing=2.5, order=5, ions=1838),
        # the largest system: 340 A, five levels, forward and adjoint
        _case("gradients_4m", "gradients", 4100000, 340.0, spacing=1.5, levels=5, order=5, ions=7100),
        # sampling: 64 independent boxes of 5,000 to 50,000 atoms, forward and
        # adjoint, replayed from one graph
        _case("replicas_64", "replicas", 5000, 0.0, replicas=64, most=50000),
        # double precision, as a program takes it to check a model or a
        # parameter set: the open droplet ...
        _case("forces_open_3k_fp64", "forces", 3000, 30.0, precision="fp64", periodic=False, cutoff=12.0, spacing=2.5,
              splitting=1),
        # ... gradients for finite-difference checks ...
        _case("gradients_23k_fp64", "gradients", 23558, 62.2, precision="fp64", ions=2),
        # ... and the benchmark system's reference
        _case("forces_1m_fp64", "forces", 1066628, 216.8, precision="fp64", cutoff=12.0, spacing=2.5, order=5,
              ions=1838),
        # molecular dynamics of a plasma in double precision: the trajectory that
        # coarse propagators are compared with
        _case("dynamics_2k_fp64", "dynamics", 2000, 38.0, precision="fp64", cutoff=8.0, steps=20),
    ]


def draw(rng):
    def between(lo, hi):  # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["forces"] * 4 + ["gradients"] * 3 + ["replicas", "dynamics"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    cutoff, spacing = rng.choice([(8.0, 1.5), (9.0, 2.0), (10.0, 2.0), (10.0, 1.7), (12.0, 2.5)])
    order, splitting = rng.choice([3, 3, 5]), rng.choice([1, 2, 2, 3])
    if what == "replicas":
        return _case("", what, between(4000, 8000), 0.0, cutoff=10.0, spacing=2.0, order=order, splitting=splitting,
                     replicas=rng.randint(5, 61), most=between(12000, 50000))
    if what == "dynamics":
        n = between(1000, 4000)
        edge = round((n / 0.0364) ** (1.0 / 3.0), 1)
        return _case("", what, n, edge, precision="fp64", cutoff=8.0, steps=rng.randint(16, 24))
    periodic = rng.random() < 0.75
    n = between(2500, 700000 if precision == "mixed" else 400000)
    if not periodic:
        n = min(n, 60000)
    edge = (n / DENSITY) ** (1.0 / 3.0)
    if periodic and edge < 2.7 * cutoff:
        cutoff, spacing = 8.0, 1.5
    stretch = [1.0] * 3
    if edge > 3.2 * cutoff:  # unequal edges where the box leaves room for them
        stretch = [rng.uniform(0.92, 1.1) for _ in range(3)]
    s = (stretch[0] * stretch[1] * stretch[2]) ** (1.0 / 3.0)
    box = tuple(round(edge * t / s, 1) for t in stretch)
    return _case("", what, n, box, precision=precision, periodic=periodic, cutoff=cutoff, spacing=spacing, order=order,
                 splitting=splitting, ions=between(2, max(4, n // 600)))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _sites(g, n, box, margin):
    """n points on a jittered lattice (a random subset of its nodes), at least
    SPACING_OF_SITES apart; with a margin they keep off the faces."""
    span = [b - 2 * margin for b in box]
    pitch = (span[0] * span[1] * span[2] / n) ** (1.0 / 3.0)
    m = [max(1, int(s / pitch)) for s in span]
    while m[0] * m[1] * m[2] < n:
        m[max(range(3), key=lambda d: span[d] / m[d])] += 1
    step = [s / k for s, k in zip(span, m)]
    node = torch.randperm(m[0] * m[1] * m[2], generator=g, device=DEV)[:n]
    ijk = torch.stack([node % m[0], (node // m[0]) % m[1], node // (m[0] * m[1])], 1).double()
    jitter = max(0.0, min(0.25, 0.499 * (min(step) - SPACING_OF_SITES)))
    u = torch.rand(n, 3, generator=g, device=DEV, dtype=torch.float64)
    return margin + (ijk + 0.5) * torch.tensor(step, device=DEV, dtype=torch.float64) + (2 * u - 1) * jitter


def _water(g, atoms, ions, box, periodic):
    """atoms - ions atoms of rigid water (the last molecules may lack hydrogens
    where the count is no multiple of three) and ions of +-1 e, the order of
    the molecules random in space."""
    ions += (atoms - ions) % 3
    waters = (atoms - ions) // 3
    sites = _sites(g, waters + ions, box, 0.0 if periodic else 0.9573)
    half, r = math.radians(104.52) / 2, 0.9572
    v = torch.randn(waters, 2, 3, generator=g, device=DEV, dtype=torch.float64)
    a = torch.nn.functional.normalize(v[:, 0], dim=1)
    b = v[:, 1] - (v[:, 1] * a).sum(1, keepdim=True) * a
    b = torch.nn.functional.normalize(b, dim=1)
    oxygen = sites[:waters]
    h1 = oxygen + r * (math.cos(half) * a + math.sin(half) * b)
    h2 = oxygen + r * (math.cos(half) * a - math.sin(half) * b)
    pos = torch.cat([torch.stack([oxygen, h1, h2], 1).reshape(-1, 3), sites[waters:]])
    q = torch.empty(len(pos), device=DEV, dtype=torch.float64)
    q[0:3 * waters:3], q[1:3 * waters:3], q[2:3 * waters:3] = -0.834, 0.417, 0.417
    q[3 * waters:] = 1.0 - 2.0 * (torch.arange(ions, device=DEV) % 2).double()
    return _inside(pos, box, periodic), q


def _inside(pos, box, periodic):
    edges = torch.tensor(box, device=DEV, dtype=torch.float64)
    if periodic:
        pos = torch.remainder(pos, edges)
        return torch.where(pos >= edges, pos - edges, pos)
    return pos.clamp(min=0.0).minimum(edges)


def _box(c):
    return (c["lx"], c["ly"], c["lz"])


def _systems(c, seed):
    """[(box, pos, q)] of the case in FP64: one system, or the replicas."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    if c["what"] != "replicas":
        return [(_box(c),) + _water(g, c["atoms"], c["ions"], _box(c), c["periodic"])]
    got, n = [], c["replicas"]
    for k in range(n):  # log-uniform sizes in a scrambled order, multiples of three
        x = ((k * 0.6180339887498949) % 1.0)
        atoms = 3 * int(round(math.exp(math.log(c["atoms"]) + x * math.log(c["most"] / c["atoms"])) / 3.0))
        box = ((atoms / DENSITY) ** (1.0 / 3.0),) * 3
        got.append((box,) + _water(g, atoms, 0, box, True))
    return got


def _plasma(c, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    pos = _inside(_sites(g, c["atoms"], _box(c), 0.0), _box(c), True)
    q = torch.ones(c["atoms"], device=DEV, dtype=torch.float64)
    vel = math.sqrt(0.05) * torch.randn(c["atoms"], 3, generator=g, device=DEV, dtype=torch.float64)
    return pos, q, vel - vel.mean(0)


def _plan(c, box, atoms):
    return MSM(box=box, periodic=c["periodic"], cutoff=c["cutoff"], spacing=c["spacing"], levels=c["levels"],
               order=c["order"], splitting=c["splitting"], precision=c["precision"], max_atoms=atoms)


TIME_STEP = 0.05


def prepare(case, seed):
    c = case
    if c["what"] == "dynamics":
        pos, q, vel = _plasma(c, seed)
        plan = _plan(c, _box(c), c["atoms"])
        _, _, force = plan.eval(pos, q, want_phi=False)
        return dict(what=c["what"], plan=plan, pos=pos, q=q, vel=vel, force=force, inv_mass=torch.ones_like(q),
                    steps=c["steps"])
    systems = _systems(c, seed)
    if c["what"] == "replicas":
        counts = [len(q) for _, _, q in systems]
        pos, q = torch.cat([p for _, p, _ in systems]), torch.cat([q for _, _, q in systems])
        batch = MSMBatch([_plan(c, box, n) for (box, _, _), n in zip(systems, counts)])
        energy = torch.empty(len(counts), device=DEV, dtype=torch.float64)
        out = [energy, torch.empty_like(q), torch.empty_like(pos), torch.empty_like(pos), torch.empty_like(q)]
        graph = batch.graph(pos, q, counts, out[0], out[1], out[2], torch.ones_like(energy), out[3], out[4])
        return dict(what=c["what"], graph=graph, out=out)
    box, pos, q = systems[0]
    kind = torch.float32 if c["precision"] == "mixed" else torch.float64
    s = dict(what=c["what"], plan=_plan(c, box, c["atoms"]), pos=pos.to(kind), q=q.to(kind))
    if c["what"] == "gradients":
        s["pos"].requires_grad_(True)
        s["q"].requires_grad_(True)
    return s


def run(state):
    s = state
    if s["what"] == "forces":
        energy, phi, force = s["plan"].eval(s["pos"], s["q"])
        return dict(energy=energy.to(phi.dtype), phi=phi, force=force)
    if s["what"] == "gradients":
        energy = MSMEnergy.apply(s["pos"], s["q"], s["plan"])
        grad_pos, grad_q = torch.autograd.grad(energy, (s["pos"], s["q"]))
        return dict(energy=energy.detach().to(grad_q.dtype), grad_pos=grad_pos, grad_q=grad_q)
    if s["what"] == "replicas":
        s["graph"].launch()
        return dict(zip(("energy", "phi", "force", "grad_pos", "grad_q"), (t.float() for t in s["out"])))
    # a trajectory from the stored configuration
    pos, vel, force = s["pos"].clone(), s["vel"].clone(), s["force"].clone()
    force, records = s["plan"].md_run(pos, vel, s["inv_mass"], s["q"], TIME_STEP, s["steps"], force=force)
    return dict(pos=pos, vel=vel, force=force, records=records)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def work(case):
    c = case
    wide = 8 if c["precision"] == "fp64" else 4
    if c["what"] == "replicas":
        systems = []
        for k in range(c["replicas"]):
            x = ((k * 0.6180339887498949) % 1.0)
            n = 3 * int(round(math.exp(math.log(c["atoms"]) + x * math.log(c["most"] / c["atoms"])) / 3.0))
            systems.append((n, n / DENSITY))
        wide = 8
    else:
        systems = [(c["atoms"], c["lx"] * c["ly"] * c["lz"])]
    grads = c["what"] in ("gradients", "replicas")
    flops = moved = 0.0
    for n, volume in systems:
        pairs = 0.5 * n * n / volume * 4.0 / 3.0 * math.pi * c["cutoff"] ** 3
        pairs = min(pairs, 0.5 * n * n)
        taps = (c["order"] + 1) ** 3 * n
        points = volume / c["spacing"] ** 3 * 8.0 / 7.0  # all levels
        sweep = points * (10.0 * math.log2(max(points, 2.0)) + 2.0)
        flops += 28.0 * pairs + 3.0 * taps + 8.0 * taps + sweep
        moved += wide * (4 * n + 4 * n)  # positions and charges in, potentials and forces (or gradients) out
        if grads:
            flops += 8.0 * taps + sweep
        if c["what"] == "replicas":
            moved += wide * 4 * n
    steps = c.get("steps", 1)
    if c["what"] == "dynamics":
        moved = 8 * 17 * c["atoms"]  # positions, velocities and forces in and out, masses and charges in ...
    return {"bytes": moved, "flops": flops * steps}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------

F64 = torch.float64


def _gamma(m, s):
    """Taylor smoothing of s^(-1/2) about s = 1 with m + 1 terms (s = rho^2)."""
    if m == 1:
        return 1.5 - 0.5 * s
    if m == 2:
        return 1.875 + s * (-1.25 + 0.375 * s)
    return 2.1875 + s * (-2.1875 + s * (1.3125 - 0.3125 * s))


def _dgamma(m, s):
    """d gamma / d s"""
    if m == 1:
        return torch.full_like(s, -0.5)
    if m == 2:
        return -1.25 + 0.75 * s
    return -2.1875 + s * (2.625 - 0.9375 * s)


def _soft(m, a, r):
    """gamma(r / a) / a: the smooth part of 1 / r beyond which it is 1 / r."""
    s = (r / a) ** 2
    return torch.where(s < 1.0, _gamma(m, s) / a, 1.0 / r.clamp(min=1e-300))


def _basis(order, d):
    """Phi(d) and its derivative: the C1 interpolating cubic, or quintic, piecewise polynomial."""
    x, sign = d.abs(), torch.sign(d)
    if order == 3:
        p = [1 + x * x * (-2.5 + 1.5 * x), 2 + x * (-4 + x * (2.5 - 0.5 * x))]
        dp = [x * (-5 + 4.5 * x), -4 + x * (5 - 1.5 * x)]
    else:
        u = [x, x - 1, x - 2]
        c = [[1, 0, -25 / 12, 5 / 12, 13 / 12, -5 / 12], [0, -16 / 24, 26 / 24, -1 / 24, -14 / 24, 5 / 24],
             [0, 2 / 24, -3 / 24, -1 / 24, 3 / 24, -1 / 24]]
        p = [sum(ck * u[j] ** k for k, ck in enumerate(c[j])) for j in range(3)]
        dp = [sum(k * ck * u[j] ** (k - 1) for k, ck in enumerate(c[j]) if k) for j in range(3)]
    f, df = torch.zeros_like(x), torch.zeros_like(x)
    for j in reversed(range(len(p))):
        f, df = torch.where(x <= j + 1, p[j], f), torch.where(x <= j + 1, dp[j], df)
    return f, df * sign


def _grids(c, box):
    """Finest spacings, and per level the first index and the number of points of each axis."""
    S = (c["order"] + 1) // 2
    if c["periodic"]:
        n0 = []
        for L in box:
            x = L / c["spacing"]
            if c["levels"]:
                m = 1 << (c["levels"] - 1)
                n0.append(max(1, math.ceil(x / m - 1e-12)) * m)
            else:
                n0.append(min(v for j in range(21) for v in [m << j for m in range(1, 9)] if v >= x - 1e-9))
        h, ns = [L / n for L, n in zip(box, n0)], [n0]
        while (len(ns) < c["levels"]) if c["levels"] else (max(ns[-1]) > 8 and not any(n & 1 for n in ns[-1])):
            ns.append([n // 2 for n in ns[-1]])
        return h, [[0] * 3 for _ in ns], ns
    h, lo, ns = [c["spacing"]] * 3, [[1 - S] * 3], [[int(math.floor(L / c["spacing"])) + 2 * S for L in box]]
    while not c["levels"] or len(ns) < c["levels"]:
        nlo = [-((-(a - (2 * S - 1))) // 2) for a in lo[-1]]
        nn = [(a + n - 1 + 2 * S - 1) // 2 - b + 1 for a, n, b in zip(lo[-1], ns[-1], nlo)]
        if not c["levels"] and (max(ns[-1]) <= 8 or max(nn) >= max(ns[-1])):
            break
        lo.append(nlo)
        ns.append(nn)
    return h, lo, ns


def _taps(c, h, lo, n, x, d):
    """Per support point: grid index along axis d, weight, derivative of the weight."""
    S = (c["order"] + 1) // 2
    t = x / h
    base = torch.floor(t)
    if not c["periodic"]:
        base = base.clamp(max=n - 2 * S)
    got = []
    for s in range(1 - S, S + 1):
        w, dw = _basis(c["order"], t - (base + s))
        i = (base + s).long()
        got.append((torch.remainder(i, n) if c["periodic"] else i - lo, w, dw / h))
    return got


def _transfer(c, lo_f, n_f, lo_c, n_c):
    """Matrix [n_c, n_f] of Phi((fine - 2 coarse) / 2) along one axis."""
    f = torch.arange(n_f, device=DEV, dtype=F64) + lo_f
    m = torch.zeros(n_c, n_f, device=DEV, dtype=F64)
    for i in range(n_c):
        d = f - 2 * (i + lo_c)
        shifts = range(-3, 4) if c["periodic"] else (0,)
        m[i] = sum(_basis(c["order"], (d + k * n_f) / 2)[0] for k in shifts)
    return m


def _along(mats, g):
    return torch.einsum("az,by,cx,zyx->abc", mats[2], mats[1], mats[0], g) if g.numel() < 4096 else \
        torch.tensordot(torch.einsum("by,zyx->zbx", mats[1], torch.tensordot(g, mats[0].T, 1)).permute(1, 2, 0),
                        mats[2].T, 1).permute(2, 0, 1)


def _convolve(kernel, E, g, periodic):
    """sum over taps |d| <= E of kernel[d] g[. - d]; kernel [2Ez+1, 2Ey+1, 2Ex+1] (z, y, x)."""
    n = g.shape
    size = n if periodic else tuple(a + b - 1 for a, b in zip(n, kernel.shape))
    k = torch.zeros(size, device=DEV, dtype=F64)
    i = [torch.arange(-e, e + 1, device=DEV) % s for e, s in zip(E, size)]
    at = (i[0][:, None, None] * size[1] + i[1][None, :, None]) * size[2] + i[2][None, None, :]
    k.view(-1).index_add_(0, at.reshape(-1), kernel.reshape(-1))
    u = torch.fft.irfftn(torch.fft.rfftn(g, s=size) * torch.fft.rfftn(k), s=size)
    return u[:n[0], :n[1], :n[2]]


def _periodic_coulomb(box, r):
    """Potential of a unit charge, its images and a neutralising background at r [n, 3], less 1 / r (Ewald)."""
    L = torch.tensor(box, device=DEV, dtype=F64)
    rc = min(box)
    alpha, kc = 5.9 / rc, 2 * 5.9 * 5.9 / rc
    v = torch.full((len(r),), -math.pi / (alpha ** 2 * box[0] * box[1] * box[2]), device=DEV, dtype=F64)
    im = [range(-int(math.ceil(rc / b)) - 1, int(math.ceil(rc / b)) + 2) for b in box]
    for a in im[0]:
        for b in im[1]:
            for e in im[2]:
                d = (r + torch.tensor([a, b, e], device=DEV, dtype=F64) * L).norm(dim=1)
                if a == b == e == 0:
                    v += torch.where(d > 0, -torch.erf(alpha * d) / d.clamp(min=1e-300), -2 * alpha / math.sqrt(math.pi))
                else:
                    v += torch.where(d < rc, torch.erfc(alpha * d) / d.clamp(min=1e-300), 0.0)
    km = [int(math.ceil(kc * b / (2 * math.pi))) for b in box]
    k = torch.cartesian_prod(*[torch.arange(-m, m + 1, device=DEV, dtype=F64) for m in km]) * (2 * math.pi / L)
    k2 = (k * k).sum(1)
    k, k2 = k[(k2 > 0) & (k2 <= kc * kc)], k2[(k2 > 0) & (k2 <= kc * kc)]
    w = torch.exp(-k2 / (4 * alpha * alpha)) / k2 * (4 * math.pi / (box[0] * box[1] * box[2]))
    for i in range(0, len(k), 4096):
        v += torch.cos(r @ k[i:i + 4096].T) @ w[i:i + 4096]
    return v


def _top(c, box, ht, A, q):
    """All pairs of the coarsest grid."""
    nz, ny, nx = q.shape
    if not c["periodic"]:
        E = (nz - 1, ny - 1, nx - 1)
        ax = [torch.arange(-e, e + 1, device=DEV, dtype=F64) * s for e, s in zip(E, ht[::-1])]
        r = (ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2).sqrt()
        return _convolve(_soft(c["splitting"], A, r), E, q, False)
    ax = []
    for n, s in zip((nx, ny, nz), ht):
        i = torch.arange(n, device=DEV)
        ax.append(torch.where(2 * i > n, i - n, i).double() * s)
    r = torch.stack([t.reshape(-1) for t in torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")][::-1], 1)
    v = _periodic_coulomb(box, r) + _soft(c["splitting"], A, r.norm(dim=1))
    im = [range(-int(math.ceil(A / b)) - 1, int(math.ceil(A / b)) + 2) for b in box]
    L = torch.tensor(box, device=DEV, dtype=F64)
    for a in im[0]:
        for b in im[1]:
            for e in im[2]:
                if (a, b, e) != (0, 0, 0):
                    d = (r + torch.tensor([a, b, e], device=DEV, dtype=F64) * L).norm(dim=1)
                    v -= torch.where(d < A, 1.0 / d - _gamma(c["splitting"], (d / A) ** 2) / A, 0.0)
    return torch.fft.irfftn(torch.fft.rfftn(q) * torch.fft.rfftn(v.reshape(nz, ny, nx)), s=q.shape)


def _pairs(m, a, d2, qj):
    """(q_j g*(r), q_j f(r)) with the force on i q_i sum f (r_i - r_j); zero at r = 0 and beyond a."""
    ok = (d2 < a * a) & (d2 > 0)
    d2 = torch.where(ok, d2, a * a)
    qj = torch.where(ok, qj, 0.0)
    ri = d2.rsqrt()
    s = d2 / (a * a)
    return qj * (ri - _gamma(m, s) / a), qj * (ri ** 3 + 2 / a ** 3 * _dgamma(m, s))


def _short(c, box, pos, q):
    """Short-range potentials and forces."""
    a, m, n = c["cutoff"], c["splitting"], len(q)
    L = torch.tensor(box, device=DEV, dtype=F64)
    nc = [max(1, int(b / a)) for b in box]
    if n <= 6000 or (c["periodic"] and min(nc) < 3):  # every pair, nearest image
        phi, force = torch.empty_like(q), torch.empty_like(pos)
        step = max(1, 20_000_000 // n)
        for i in range(0, n, step):
            d = pos[i:i + step, None] - pos[None]
            if c["periodic"]:
                d -= L * torch.round(d / L)
            p, f = _pairs(m, a, (d * d).sum(2), q[None])
            phi[i:i + step] = p.sum(1)
            force[i:i + step] = q[i:i + step, None] * (f[:, :, None] * d).sum(1)
        return phi, force
    w = L / torch.tensor(nc, device=DEV, dtype=F64)
    ci = (pos / w).long().minimum(torch.tensor(nc, device=DEV) - 1)
    cell = (ci[:, 2] * nc[1] + ci[:, 1]) * nc[0] + ci[:, 0]
    ncell = nc[0] * nc[1] * nc[2]
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=ncell)
    start = torch.cumsum(count, 0) - count
    most = int(count.max())
    slot = torch.full((ncell + 1, most), n, device=DEV, dtype=torch.long)  # the extra cell is empty
    slot[cell[order], torch.arange(n, device=DEV) - start[cell[order]]] = order
    P = torch.cat([pos, torch.full((1, 3), 1e9, device=DEV, dtype=F64)])
    Q = torch.cat([q, torch.zeros(1, device=DEV, dtype=F64)])
    phi, force = torch.zeros(n + 1, device=DEV, dtype=F64), torch.zeros(n + 1, 3, device=DEV, dtype=F64)
    step = max(1, 30_000_000 // (most * most))
    offsets = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    for c0 in range(0, ncell, step):
        me = torch.arange(c0, min(c0 + step, ncell), device=DEV)
        xyz = [me % nc[0], (me // nc[0]) % nc[1], me // (nc[0] * nc[1])]
        si = slot[me]
        xi = P[si]
        ph, fo = torch.zeros_like(xi[:, :, 0]), torch.zeros_like(xi)
        for o in offsets:
            at = [v + k for v, k in zip(xyz, o)]
            img = torch.stack([torch.div(v, k, rounding_mode="floor") for v, k in zip(at, nc)], 1).double()
            wrapped = [v % k for v, k in zip(at, nc)]
            nb = (wrapped[2] * nc[1] + wrapped[1]) * nc[0] + wrapped[0]
            if not c["periodic"]:
                nb = torch.where((img != 0).any(1), ncell, nb)
            sj = slot[nb]
            xj = P[sj] + (img * L)[:, None] * float(c["periodic"])
            d = [xi[:, :, None, k] - xj[:, None, :, k] for k in range(3)]
            p, f = _pairs(m, a, d[0] * d[0] + d[1] * d[1] + d[2] * d[2], Q[sj][:, None])
            ph += p.sum(2)
            for k in range(3):
                fo[:, :, k] += (f * d[k]).sum(2)
        phi[si], force[si] = ph, fo * Q[si][:, :, None]
    return phi[:n], force[:n]


def _msm(c, box, pos, q):
    """Energy, potentials and forces by MSM with the case's parameters."""
    m, a = c["splitting"], c["cutoff"]
    h, lo, ns = _grids(c, box)
    top = len(ns) - 1
    shape = [tuple(reversed(n)) for n in ns]
    taps = [_taps(c, h[d], lo[0][d], ns[0][d], pos[:, d], d) for d in range(3)]
    charge = [torch.zeros(shape[0], device=DEV, dtype=F64)]
    flat = charge[0].view(-1)
    for iz, wz, _ in taps[2]:
        for iy, wy, _ in taps[1]:
            for ix, wx, _ in taps[0]:
                flat.index_add_(0, (iz * ns[0][1] + iy) * ns[0][0] + ix, q * wz * wy * wx)
    E = [int(math.ceil(2 * a / x)) for x in h]
    ax = [torch.arange(-e, e + 1, device=DEV, dtype=F64) * x for e, x in zip(E, h)]
    r = (ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2).sqrt()
    kernel = torch.where(r < 2 * a, _soft(m, a, r) - _soft(m, 2 * a, r), 0.0)
    mats, u = [], []
    for k in range(top):
        mats.append([_transfer(c, lo[k][d], ns[k][d], lo[k + 1][d], ns[k + 1][d]) for d in range(3)])
        charge.append(_along(mats[k], charge[k]))
        u.append(0.5 ** k * _convolve(kernel, E[::-1], charge[k], c["periodic"]))
    u.append(_top(c, box, [x * 2 ** top for x in h], a * 2 ** top, charge[top]))
    for k in reversed(range(top)):
        u[k] = u[k] + _along([t.T for t in mats[k]], u[k + 1])
    flat = u[0].reshape(-1)
    phi, force = _short(c, box, pos, q)
    for iz, wz, dz in taps[2]:
        for iy, wy, dy in taps[1]:
            for ix, wx, dx in taps[0]:
                v = flat[(iz * ns[0][1] + iy) * ns[0][0] + ix]
                phi += v * wx * wy * wz
                v = v * q
                force[:, 0] -= v * dx * wy * wz
                force[:, 1] -= v * wx * dy * wz
                force[:, 2] -= v * wx * wy * dz
    phi -= q * float(_gamma(m, torch.zeros((), dtype=F64))) / a
    return 0.5 * (q * phi).sum(), phi, force


def exact(case, seed):
    c = case
    if c["what"] == "dynamics":
        pos, q, vel = _plasma(c, seed)
        L = torch.tensor(_box(c), device=DEV, dtype=F64)
        _, _, force = _msm(c, _box(c), pos, q)
        records = []
        for _ in range(c["steps"]):
            vel = vel + 0.5 * TIME_STEP * force
            pos = pos + TIME_STEP * vel
            pos = pos - L * torch.floor(pos / L)
            e, _, force = _msm(c, _box(c), pos, q)
            vel = vel + 0.5 * TIME_STEP * force
            kinetic = 0.5 * (vel * vel).sum()
            records.append(torch.cat([torch.stack([e, kinetic, e + kinetic]), vel.sum(0)]))
        return dict(pos=pos, vel=vel, force=force, records=torch.stack(records))
    # the inputs as the program holds them
    kind = torch.float32 if c["precision"] == "mixed" and c["what"] != "replicas" else F64
    got = [_msm(c, box, pos.to(kind).double(), q.to(kind).double()) for box, pos, q in _systems(c, seed)]
    if c["what"] == "forces":
        energy, phi, force = got[0]
        return dict(energy=energy, phi=phi, force=force)
    if c["what"] == "gradients":  # the energy is quadratic in the charges with a symmetric operator
        energy, phi, force = got[0]
        return dict(energy=energy, grad_pos=-force, grad_q=phi)
    energy = torch.stack([g[0] for g in got])
    phi, force = torch.cat([g[1] for g in got]), torch.cat([g[2] for g in got])
    return dict(energy=energy, phi=phi, force=force, grad_pos=-force, grad_q=phi)
