"""The work that users of this library have it do, as cases that can be timed and checked.

A particle set is a periodic box of side L = 4 n^(1/3) (about the 128^3 set's 500 / 128 per
particle) with a mesh of about n^(1/3) cells a side, r_s = 1.2 L / mesh and r_c = 4.5 r_s (the
paper's choice), holding either uniform positions or 60 % of its mass in NFW halos (concentration
10, dN/dM ~ M^-1.9, one halo per ~520 particles).  The kinds of case:

  step     a time step's short-range force: the leaf set is built on the GPU from the step's
           positions (they move every step) and the forces are summed; with "theta" the pair list
           is split and the far entries go through the multipoles; with "mesh" the long-range PM
           force is added, which makes it the whole force of a step
  forces   the force on a leaf set that is kept (several evaluations on one set of positions:
           option studies, fixed neighbour sets, the benchmark's headline)
  adjoint  gradients on a kept leaf set
  grad     forward and backward through the differentiable entry point, from positions
  pm       the long-range force alone
  batch    many small boxes in one kept leaf set, one launch
"""
import math
import random

import numpy as np
import torch

import paper_2107_14008_gb300 as psr

G = 1.0
CONC = 10.0  # NFW concentration
PRECISION = {"fp64": psr.PSR_FP64, "exact": psr.PSR_FP32_EXACT, "table": psr.PSR_FP32_TABLE}
INTERP = {"linear": psr.PSR_LINEAR, "cubic": psr.PSR_CUBIC, "taylor2": psr.PSR_TAYLOR2,
          "taylor4": psr.PSR_TAYLOR4}
DEVICE = "cuda"

# What a pair within the cutoff needs, in FP32 or FP64 operations: the difference (3), its square
# (5), 1/r (1), T by interpolation (4), the weight (3), the three sums (6); the adjoint has the
# tidal tensor applied to a vector and the mass term in place of the three sums.
PAIR_FLOPS, ADJ_FLOPS = 22, 46
# share of the pairs within the cutoff that stay with the near list of a split at theta = 0.5
NEAR_SHARE = 0.6


def _case(name, kind, n, set_, **more):
    c = {"kind": kind, "n": n, "set": set_, "masses": "equal", "max_leaf": 32, "precision": "table",
         "interp": "linear", "table_n": 0, "kahan": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest simulation step: an interactive or unit-test sized box, all latency
        _case("step_17c_uniform", "step", 17 ** 3, "uniform"),
        # the smallest workload of the benchmark, on a kept leaf set
        _case("forces_32c_uniform", "forces", 32 ** 3, "uniform"),
        # the whole force of a step, short and long range, of a small production box
        _case("step_64c_total", "step", 64 ** 3, "nfw", mesh=64),
        # the benchmark's headline: 128^3 clustered particles, kept leaf set
        _case("forces_128c_nfw", "forces", 128 ** 3, "nfw"),
        # the largest step: 256^3 clustered particles in leaves of up to 64
        _case("step_256c_nfw", "step", 256 ** 3, "nfw", max_leaf=64),
        # gradients for a fit on the differentiation workload's set
        _case("adjoint_64c_nfw", "adjoint", 64 ** 3, "nfw"),
        # forward + backward from positions: ragged count, particles of two masses
        _case("grad_500009_two_masses", "grad", 500009, "nfw", masses="two"),
        # a step with the multipole split of the short range, order 4
        _case("step_128c_split", "step", 128 ** 3, "nfw", theta=0.5, order=4),
        # the long-range force alone on the headline's set
        _case("pm_128c", "pm", 128 ** 3, "nfw", mesh=128),
        # double precision: reference forces for validating the FP32 path
        _case("forces_48c_fp64", "forces", 48 ** 3, "nfw", precision="fp64"),
        # double precision gradients, as finite-difference checks and optimisers take them
        _case("adjoint_32c_fp64", "adjoint", 32 ** 3, "uniform", precision="fp64"),
        # 64 independent boxes of 8^3 to 64^3 particles in one launch
        _case("batch_64_boxes", "batch", 64, "mixed"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "forces", "forces", "forces", "adjoint", "adjoint",
                       "grad", "pm", "batch"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    set_ = rng.choice(["uniform", "nfw", "nfw"])
    more = {"masses": rng.choice(["equal", "equal", "two"]), "max_leaf": rng.choice([16, 32, 32, 64])}
    if kind == "batch":
        return _case(None, "batch", rng.randint(4, 64), "mixed", max_leaf=rng.choice([16, 32]))
    if kind == "pm":
        n = size(30 ** 3, 160 ** 3)
        return _case(None, "pm", n, set_, masses=more["masses"], mesh=_mesh(n))
    if kind == "grad":
        return _case(None, "grad", size(16 ** 3, 100 ** 3), set_, **more)
    if kind == "step":
        n = size(15 ** 3, 160 ** 3)
        form = rng.choice(["plain", "plain", "total", "split"])
        if form == "total":
            more["mesh"] = _mesh(n)
        if form == "split":
            n = size(40 ** 3, 130 ** 3)
            more.update(theta=rng.choice([0.5, 0.7]), order=rng.choice([4, 4, 6]))
        return _case(None, "step", n, set_, **more)
    arith = rng.choice(["table", "table", "table", "exact", "fp64"])
    if arith == "fp64":
        n = size(16 ** 3, 48 ** 3 if kind == "forces" else 36 ** 3)
        more.update(precision="fp64")
        if kind == "forces":
            more["interp"] = rng.choice(["linear", "taylor4"])
    elif arith == "exact":
        n = size(20 ** 3, 80 ** 3)
        more.update(precision="exact", kahan=rng.random() < 0.3)
    else:
        n = size(20 ** 3, 130 ** 3)
        interp = rng.choice(["linear", "linear", "cubic"] + (["taylor2"] if kind == "forces" else []))
        more.update(interp=interp, kahan=rng.random() < 0.3,
                    table_n=rng.choice([0, 4096]) if interp == "linear" else 0)
    return _case(None, kind, n, set_, **more)


# ------------------------------------------------------------------ inputs --
def _mesh(n):
    """Mesh cells a side for n particles: about one particle a cell, even, at least 8."""
    return max(8, 2 * int(round(0.5 * n ** (1.0 / 3.0))))


def _side(n):
    return 4.0 * n ** (1.0 / 3.0)


def _box(case, n=None):
    n = case["n"] if n is None else n
    L = _side(n)
    r_s = 1.2 * L / (case.get("mesh") or _mesh(n))
    return L, r_s, 4.5 * r_s


def _nfw_table():
    """Quantiles of the NFW enclosed mass out to the concentration, in scale radii."""
    s = np.linspace(0.0, 1.0, 1 << 16) ** 2 * CONC
    mu = np.log1p(s) - s / (1.0 + s)
    u = np.linspace(0.0, 1.0, 1 << 14)
    return np.interp(u * mu[-1], mu, s)


def _halo_counts(n, rng):
    """Particles of each halo, and how many in all."""
    k = max(1, int(round(n * 4000 / 128 ** 3)))
    lo, hi, a = 1e-5, 1e-2, -0.9
    m = (lo ** a + rng.random(k) * (hi ** a - lo ** a)) ** (1.0 / a)
    return np.floor(m * (0.6 * n / m.sum())).astype(np.int64)


def _positions(n, L, set_, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)

    def rand(*shape):
        return torch.rand(*shape, dtype=torch.float64, device=DEVICE, generator=gen)

    pos = rand(n, 3) * L
    if set_ == "nfw":
        counts = _halo_counts(n, np.random.default_rng(seed))
        k, nh = len(counts), int(counts.sum())
        c = torch.from_numpy(counts).to(DEVICE)
        halo = torch.repeat_interleave(torch.arange(k, device=DEVICE), c, output_size=nh)
        r200 = (3.0 * c / n * L ** 3 / (4.0 * math.pi * 200.0)) ** (1.0 / 3.0)
        table = torch.from_numpy(_nfw_table()).to(DEVICE)
        u = rand(nh) * (table.numel() - 1)
        i = u.long().clamp(max=table.numel() - 2)
        s = torch.lerp(table[i], table[i + 1], u - i)
        cz, phi = 2.0 * rand(nh) - 1.0, 2.0 * math.pi * rand(nh)
        sz = (1.0 - cz * cz).clamp(min=0.0).sqrt()
        d = torch.stack([sz * phi.cos(), sz * phi.sin(), cz], 1)
        pos[:nh] = (rand(k, 3) * L)[halo] + d * (s * r200[halo] / CONC)[:, None]
        pos = pos[torch.randperm(n, device=DEVICE, generator=gen)]  # a catalogue's order
    pos = torch.remainder(pos, L)
    return torch.where(pos >= L, torch.zeros_like(pos), pos).contiguous()


def _masses(n, kind, seed):
    m = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEVICE)
    if kind == "two":  # two species, one five times the other's mass
        gen = torch.Generator(device=DEVICE)
        gen.manual_seed(seed + 7)
        m = m * torch.where(torch.rand(n, device=DEVICE, generator=gen) < 0.2, 5.0 / 1.8, 1.0 / 1.8)
    return m


def _cotangent(n, dtype, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed + 11)
    return torch.randn(n, 3, dtype=dtype, device=DEVICE, generator=gen)


def _options(case):
    return psr.Options(precision=PRECISION[case["precision"]], interp=INTERP[case["interp"]],
                       table_n=case["table_n"],
                       accum=psr.PSR_ACC_KAHAN32 if case["kahan"] else psr.PSR_ACC_FP64)


def _batch_sizes(case):
    """Particle counts of a batch's boxes, 8^3 to 64^3."""
    rng = random.Random(case["n"])
    return [int(round(math.exp(rng.uniform(math.log(8 ** 3), math.log(64 ** 3)))))
            for _ in range(case["n"])]


def _batch_boxes(case, seed):
    out = []
    for b, n in enumerate(_batch_sizes(case)):
        L, r_s, r_c = _box(case, n)
        pos = _positions(n, L, "nfw" if b % 2 else "uniform", seed * 1000 + b)
        out.append((pos, torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEVICE), L, r_s, r_c))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "opts": _options(case)}
    if kind == "batch":
        boxes = [(p.cpu().numpy(), m.cpu().numpy(), L, r_s, r_c, G)
                 for p, m, L, r_s, r_c in _batch_boxes(case, seed)]
        s["leaves"] = psr.Leaves.build_batch(boxes, max_leaf=case["max_leaf"]).upload(DEVICE)
        return s
    L, r_s, r_c = _box(case)
    s["box"] = (L, r_s, r_c)
    s["pos"] = _positions(case["n"], L, case["set"], seed)
    s["mass"] = _masses(case["n"], case["masses"], seed)
    fp64 = case["precision"] == "fp64"
    if case.get("mesh"):
        s["pm"] = psr.PM(case["mesh"], device=DEVICE)
    if kind in ("forces", "adjoint"):
        s["leaves"] = psr.Leaves.device_build(s["pos"], s["mass"], L, r_s, r_c, G,
                                              max_leaf=case["max_leaf"], fp64=fp64)
    if kind in ("adjoint", "grad"):
        s["cot"] = _cotangent(case["n"], torch.float64 if fp64 or kind == "grad" else torch.float32, seed)
    return s


def run(s):
    case, kind, opts = s["case"], s["case"]["kind"], s["opts"]
    if kind in ("forces", "batch"):
        return s["leaves"].forces(opts)
    if kind == "adjoint":
        gx, gm = s["leaves"].adjoint(s["cot"], opts)
        return {"grad_pos": gx, "grad_mass": gm}
    L, r_s, r_c = s["box"]
    if kind == "pm":
        return s["pm"].forces(s["pos"], s["mass"], L, r_s, G)
    if kind == "grad":
        pos, mass = s["pos"].detach().requires_grad_(), s["mass"].detach().requires_grad_()
        acc = psr.forces(pos, mass, L, r_s, r_c, G, opts, case["max_leaf"])
        gx, gm = torch.autograd.grad(acc, (pos, mass), s["cot"])
        return {"acc": acc.detach(), "grad_pos": gx, "grad_mass": gm}
    if case.get("theta"):
        lv = psr.Leaves.device_build(s["pos"], s["mass"], L, r_s, r_c, G,
                                     max_leaf=case["max_leaf"], theta=case["theta"])
        acc = lv.forces(opts)
        return lv.fmm_forces(case["order"], out=acc, accumulate=True)
    lv = psr.Leaves.device_build(s["pos"], s["mass"], L, r_s, r_c, G, max_leaf=case["max_leaf"],
                                 fp64=False)
    acc = lv.forces(opts)
    if "pm" in s:
        s["pm"].forces(s["pos"], s["mass"], L, r_s, G, out=acc, accumulate=True)
    return acc


# -------------------------------------------------------------------- work --
def _pairs(n, set_, r_c, L):
    """Pairs within the cutoff, to some per cent: the uniform background's, and those inside the
    halos (whose diameters are mostly below the cutoff)."""
    p = n * n * (4.0 / 3.0) * math.pi * (r_c / L) ** 3
    if set_ == "nfw":
        p += float((_halo_counts(n, np.random.default_rng(0)).astype(np.float64) ** 2).sum())
    return p


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        pairs = sum(_pairs(m, "nfw" if b % 2 else "uniform", *(_box(case, m)[2::-2]))
                    for b, m in enumerate(sizes))
        return {"bytes": 28.0 * sum(sizes), "flops": PAIR_FLOPS * pairs}
    L, _, r_c = _box(case)
    pairs = _pairs(n, case["set"], r_c, L)
    wide = 2.0 if case["precision"] == "fp64" else 1.0
    mesh = float(case.get("mesh") or 0) ** 3
    # deposit and three interpolations of 8 points, and four real transforms
    pm = n * 8 * 9 + 4 * 2.5 * mesh * math.log2(mesh) if mesh else 0.0
    if kind == "pm":
        return {"bytes": 44.0 * n, "flops": pm}
    if kind == "forces":
        return {"bytes": wide * 28.0 * n, "flops": PAIR_FLOPS * pairs}
    if kind == "adjoint":
        return {"bytes": wide * 44.0 * n, "flops": ADJ_FLOPS * pairs}
    if kind == "grad":
        return {"bytes": 112.0 * n, "flops": (PAIR_FLOPS + ADJ_FLOPS) * pairs}
    near = NEAR_SHARE if case.get("theta") else 1.0
    return {"bytes": 44.0 * n, "flops": near * PAIR_FLOPS * pairs + pm}


# ------------------------------------------------- the same in 64 bits, plainly --
def _pair_blocks(pos, L, r_c):
    """(order, blocks): particles sorted by cell, and for runs of sorted targets the pairs with
    0 < r < r_c as (first target, counts per target, target, source, difference)."""
    n, dev = pos.shape[0], pos.device
    nc = max(1, int(3.0 * L / r_c))
    while nc > 1 and nc ** 3 > 8 * n:
        nc -= 1
    h = L / nc
    cell = (pos / h).long().clamp(max=nc - 1)
    key = (cell[:, 0] * nc + cell[:, 1]) * nc + cell[:, 2]
    key, order = torch.sort(key)
    p, cell = pos[order].contiguous(), cell[order]
    start = torch.searchsorted(key, torch.arange(nc ** 3 + 1, device=dev))
    reach = int(math.ceil(r_c / h))
    cols = []
    for a in range(-reach, reach + 1):
        for b in range(-reach, reach + 1):
            g2 = (max(abs(a) - 1, 0) * h) ** 2 + (max(abs(b) - 1, 0) * h) ** 2
            if g2 < r_c * r_c:
                cols.append((a, b, int(math.ceil(math.sqrt(r_c * r_c - g2) / h))))
    images = range(-((reach + nc - 1) // nc), (reach + nc - 1) // nc + 1)
    ca = torch.tensor([(a, b, z, k) for a, b, z in cols for k in images], device=dev)
    m = ca.shape[0]

    def ranges(t0, t1):
        c = cell[t0:t1, None, :]
        x, y = c[..., 0] + ca[:, 0], c[..., 1] + ca[:, 1]
        z0 = torch.maximum(c[..., 2] - ca[:, 2], ca[:, 3] * nc)
        z1 = torch.minimum(c[..., 2] + ca[:, 2], ca[:, 3] * nc + nc - 1)
        ok = z0 <= z1
        row = (torch.remainder(x, nc) * nc + torch.remainder(y, nc)) * nc
        zk = (ca[:, 3] * nc).expand_as(z0)
        lo = start[torch.where(ok, row + z0 - zk, 0)]
        hi = start[torch.where(ok, row + z1 - zk + 1, 0)]
        im = torch.stack([torch.div(x, nc, rounding_mode="floor"),
                          torch.div(y, nc, rounding_mode="floor"), ca[:, 3].expand_as(x)], -1)
        return lo, hi - lo, im

    def blocks():
        piece = 1 << 14
        for q0 in range(0, n, piece):
            q1 = min(n, q0 + piece)
            lo, cnt, im = ranges(q0, q1)
            per = torch.cumsum(cnt.sum(1), 0).cpu().numpy()
            t0 = q0
            while t0 < q1:  # as many targets as stay below 100 million candidates
                base = per[t0 - q0 - 1] if t0 > q0 else 0
                t1 = q0 + max(int(np.searchsorted(per, base + 100_000_000, side="right")), t0 - q0 + 1)
                t1 = min(t1, q1)
                c = cnt[t0 - q0:t1 - q0].reshape(-1)
                total = int(c.sum())
                if total:
                    rid = torch.repeat_interleave(torch.arange(c.numel(), device=dev), c, output_size=total)
                    off = lo[t0 - q0:t1 - q0].reshape(-1) - (torch.cumsum(c, 0) - c)
                    src = torch.arange(total, device=dev) + off[rid]
                    tgt = torch.div(rid, m, rounding_mode="floor")
                    sh = im[t0 - q0:t1 - q0].reshape(-1, 3).double() * L
                    d = p[src] + sh[rid] - p[t0 + tgt]
                    r2 = (d * d).sum(1)
                    keep = ((r2 > 0) & (r2 < r_c * r_c)).nonzero()[:, 0]
                    tgt, src, d = tgt[keep], src[keep], d[keep]
                    yield t0, torch.bincount(tgt, minlength=t1 - t0), t0 + tgt, src, d
                t0 = t1

    return order, blocks()


def _weights(d, r_s):
    """x = r / 2 r_s, T(x), 1/r and exp(-x^2) of the pair differences."""
    r = d.square().sum(1).sqrt()
    x = r / (2.0 * r_s)
    e = torch.exp(-x * x)
    return x, torch.erfc(x) + (2.0 / math.sqrt(math.pi)) * x * e, 1.0 / r, e


def _sums(values, counts):
    return torch.segment_reduce(values, "sum", lengths=counts, axis=0, unsafe=True)


def _forces64(pos, mass, L, r_s, r_c):
    order, blocks = _pair_blocks(pos, L, r_c)
    m = mass[order]
    acc = torch.zeros(pos.shape[0], 3, dtype=torch.float64, device=pos.device)
    for t0, counts, _, src, d in blocks:
        _, T, ri, _ = _weights(d, r_s)
        acc[order[t0:t0 + counts.numel()]] = G * _sums(d * (m[src] * T * ri ** 3)[:, None], counts)
    return acc


def _gradients64(pos, mass, cot, L, r_s, r_c):
    order, blocks = _pair_blocks(pos, L, r_c)
    m, c = mass[order], cot[order]
    gx = torch.zeros(pos.shape[0], 3, dtype=torch.float64, device=pos.device)
    gm = torch.zeros(pos.shape[0], dtype=torch.float64, device=pos.device)
    for t0, counts, tgt, src, d in blocks:
        _, T, ri, e = _weights(d, r_s)
        g = T * ri ** 3
        # g'(r)/r
        h = -3.0 * g * ri ** 2 - e * ri ** 2 / (2.0 * math.sqrt(math.pi) * r_s ** 3)
        v = m[tgt, None] * c[src] - m[src, None] * c[tgt]
        at = order[t0:t0 + counts.numel()]
        gx[at] = G * _sums(g[:, None] * v + (h * (d * v).sum(1))[:, None] * d, counts)
        gm[at] = -G * _sums(g * (d * c[src]).sum(1), counts)
    return gx, gm


def _mesh64(pos, mass, L, r_s, N):
    """The mesh method: cloud-in-cell, filtered Green's function, spectral gradient."""
    dev = pos.device
    u = pos * (N / L)
    i0 = u.floor().clamp(max=N - 1)
    f = u - i0
    i0 = i0.long()
    corners = []
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                ix, iy, iz = ((i0[:, q] + s) % N for q, s in enumerate((a, b, c)))
                w = torch.ones_like(f[:, 0])
                for q, s in enumerate((a, b, c)):
                    w = w * (f[:, q] if s else 1.0 - f[:, q])
                corners.append(((ix * N + iy) * N + iz, w))
    rho = torch.zeros(N ** 3, dtype=torch.float64, device=dev)
    for at, w in corners:
        rho.index_add_(0, at, w * mass)
    k1 = 2.0 * math.pi / L * torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=dev)
    kz = 2.0 * math.pi / L * torch.arange(N // 2 + 1, dtype=torch.float64, device=dev)
    ks = (k1[:, None, None], k1[None, :, None], kz[None, None, :])
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    green = -4.0 * math.pi * G * torch.exp(-k2 * r_s ** 2) / k2.clamp(min=1e-300)
    for k in ks:
        green = green / torch.sinc(k * (0.5 * L / N) / math.pi) ** 4
    green[0, 0, 0] = 0.0
    phi = torch.fft.rfftn(rho.reshape(N, N, N) / (L / N) ** 3) * green
    acc = torch.zeros_like(pos)
    for q, k in enumerate(ks):
        k = k.clone()
        k.view(-1)[N // 2] = 0.0
        g = torch.fft.irfftn(-1j * k * phi, s=(N, N, N)).reshape(-1)
        for at, w in corners:
            acc[:, q] += w * g[at]
    return acc


def exact(case, seed):
    """run()'s outputs in 64 bits by plain torch (with the split: the sum the multipoles expand)."""
    kind = case["kind"]
    if kind == "batch":
        boxes = _batch_boxes(case, seed)
        return torch.cat([_forces64(p, m, L, r_s, r_c) for p, m, L, r_s, r_c in boxes])
    L, r_s, r_c = _box(case)
    if _pairs(case["n"], case["set"], r_c, L) > 1.5e10:
        return None  # minutes of pair sums
    pos = _positions(case["n"], L, case["set"], seed)
    mass = _masses(case["n"], case["masses"], seed)
    if kind == "pm":
        return _mesh64(pos, mass, L, r_s, case["mesh"])
    if kind in ("adjoint", "grad"):
        cot = _cotangent(case["n"], torch.float64 if case["precision"] == "fp64" or kind == "grad"
                         else torch.float32, seed).double()
        gx, gm = _gradients64(pos, mass, cot, L, r_s, r_c)
        out = {"grad_pos": gx, "grad_mass": gm}
        if kind == "grad":
            out["acc"] = _forces64(pos, mass, L, r_s, r_c)
        return out
    acc = _forces64(pos, mass, L, r_s, r_c)
    if case.get("mesh"):
        acc = acc + _mesh64(pos, mass, L, r_s, case["mesh"])
    return acc
