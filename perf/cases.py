"""Performance cases of libusr: what a program that uses the library has it do, through its public entry points.

One pass is one evaluation as a simulation step makes it: the force on and the potential at every charge of one
periodic system, or of a batch of systems for the serving loop (the steps between two reports, which ask for no
energy).  `prepare` makes what a program holds before it: charges in device or pinned host memory and a context (or
a server), both kept over many evaluations.

Systems: `water` is the serving stream's generator (rigid 3-site waters, 0.1 charges per cubic Angstrom); `slab` is a
membrane-shaped box (chains of 12 charged beads between two water layers); `ions` are random charges of a hard-core
liquid in a box with no equal sides.  Forms (convolution arithmetic, spreading stencil, width in grid spacings):
`tight` FP32 / 12 / 1.0 (the library's defaults), `serving` TF32x3 / 10 / 0.9, `fast` BF16x3 / 8 / 0.83.
"""
import math

import numpy as np
import torch

from paper_1911_01377_gb300 import usr
from paper_1911_01377_gb300 import workloads as W
from paper_1911_01377_gb300.autograd import usr_energy

FORMS = {"tight": (0, 12, 1.0), "serving": (1, 10, 0.9), "fast": (2, 8, 0.83)}
# entry: "device" usr_eval on device buffers, "host" usr_eval_host from and to pinned host memory, "grad" usr_energy
# and its gradients, "server" Server.submit / wait / poll
DENSITY = 0.1


def _case(name, entry, system, n, box, grid, r_c, form, multilevel=0):
    return {"name": name, "entry": entry, "system": system, "n": n, "lx": box[0], "ly": box[1], "lz": box[2],
            "gx": grid[0], "gy": grid[1], "gz": grid[2], "r_c": r_c, "form": form, "multilevel": multilevel}


def _cube(n):
    L = (n / DENSITY) ** (1.0 / 3.0)
    return (L, L, L)


def listed():
    return [
        # the smallest request of a serving stream: a small solvated molecule, for a program on the host
        _case("water_2k_host", "host", "water", 2001, _cube(2001), (24, 24, 24), 9.0, "serving"),
        # a small simulation box in the default (tight) form
        _case("water_3k", "device", "water", 3000, (31.0,) * 3, (32, 32, 32), 9.0, "tight"),
        # ragged box and grid, no size a multiple of anything: only the FP32 form takes it
        _case("ions_7k_ragged", "device", "ions", 7013, (47.9, 36.1, 52.7), (47, 35, 53), 8.5, "tight"),
        # a differentiable program: the energy's gradients in positions and charges
        _case("water_20k_grad", "grad", "water", 20001, (58.5,) * 3, (48, 48, 48), 9.0, "serving"),
        # the membrane benchmark at the ends of its cutoff range, in its timed form
        _case("slab_64k_rc8", "device", "slab", 63996, (80.0, 80.0, 100.0), (64, 64, 80), 8.0, "fast"),
        _case("slab_64k_rc13", "device", "slab", 63996, (80.0, 80.0, 100.0), (64, 64, 80), 13.0, "fast"),
        # the same membrane in the tight form
        _case("slab_64k_tight", "device", "slab", 63996, (80.0, 80.0, 100.0), (64, 64, 80), 10.0, "tight"),
        # 24 systems of a serving stream at once, 2 k to 60 k charges each
        _case("serving_24", "server", "water", 24, (0.0,) * 3, (0, 0, 0), 9.0, "serving"),
        # the largest request of a serving stream, from and to host memory
        _case("water_200k_host", "host", "water", 199998, _cube(199998), (128, 128, 128), 9.0, "serving"),
        # a large box whose wide terms go to the coarse grid
        _case("water_200k_multilevel", "device", "water", 199998, _cube(199998), (128, 128, 128), 9.0, "serving",
              multilevel=1),
        # the largest single system
        _case("water_1m", "device", "water", 1064799, (220.0,) * 3, (176, 176, 176), 10.0, "fast", multilevel=1),
    ]


def _axis_grid(L, spacing, multiple, at_least):
    return max(at_least, int(round(L / spacing / multiple)) * multiple)


def draw(rng):
    """One more case: any entry, system and form, charges over the whole range on a logarithmic scale, cutoffs from
    8 to 13 Angstrom where the box allows them, grids from 1 to 1.3 Angstrom (odd ones in the FP32 form).  The fast
    form takes the wide terms of waters, and of everything beyond 70 k charges, to the coarse grid, as a user who
    needs the potential's fifth digit does."""
    entry = rng.choice(("device", "device", "device", "device", "host", "host", "grad", "server"))
    if entry == "server":
        c = _case("", entry, "water", rng.randint(6, 24), (0.0,) * 3, (0,) * 3, 9.0, "serving")
        del c["name"]
        return c
    form = rng.choice(("tight", "serving", "fast"))
    system = rng.choice(("water", "water", "ions", "slab"))
    n_max = {"tight": 150000, "serving": 300000, "fast": 500000}[form]
    n = int(math.exp(rng.uniform(math.log(2000 if (form, system) != ("fast", "water") else 10000), math.log(n_max))))
    n = 3 * (n // 3) + (0 if system == "water" else rng.randint(0, 2))
    vol = n / DENSITY
    if system == "water":
        box = _cube(n)
    else:
        ax, ay = rng.uniform(0.85, 1.2), rng.uniform(0.85, 1.2)
        L = vol ** (1.0 / 3.0)
        box = (ax * L, ay * L, L / (ax * ay))
    r_max = min(13.0, min(box) / 3.001)
    r_c = round(rng.uniform(min(8.0, r_max), r_max), 3)
    spacing = rng.uniform(1.0, 1.3)
    mult = {"tight": 1, "serving": 4, "fast": 8}[form]
    multilevel = int((form == "fast" and (system == "water" or n > 70000)) or
                     (form == "serving" and n > 50000 and rng.random() < 0.3))
    if multilevel:
        mult = 8
    grid = tuple(_axis_grid(b, spacing, mult, 40 if multilevel else 24) for b in box)
    c = _case("", entry, system, n, box, grid, r_c, form, multilevel)
    del c["name"]
    try:
        usr.usr_plan(usr.make_params(box, grid, r_c, "C1_B2", max_atoms=n, **_kw(c)))
    except usr.UsrError:
        return draw(rng)        # cells of more points than a spreading tile holds (large cutoffs on few cells)
    return c


# ---------------------------------------------------------------- inputs

def _water(seed, n, box):
    """Waters at the box's own size (the generator's density may differ from the box by a little): (n, 4)."""
    b, rows = W.lattice_water_box(seed, n, n / (box[0] * box[1] * box[2]))
    return rows


def _ions(seed, n, box):
    """n random charges (normal, unit variance, neutral) on a jittered lattice: no two closer than 1.2 Angstrom."""
    r = np.random.default_rng(seed)
    box = np.asarray(box)
    a = (box.prod() / n) ** (1.0 / 3.0)
    m = np.floor(box / a).astype(np.int64)
    while m.prod() < n:
        m[np.argmax(box / m)] += 1
    site = r.permutation(int(m.prod()))[:n]
    ijk = np.stack([site % m[0], site // m[0] % m[1], site // (m[0] * m[1])], axis=1)
    step = box / m
    jit = np.maximum(0.0, 0.5 * (step - 1.2))
    xyz = (ijk + 0.5) * step + r.uniform(-1.0, 1.0, (n, 3)) * jit
    q = r.normal(0.0, 1.0, n)
    return np.concatenate([xyz, (q - q.mean())[:, None]], axis=1).astype(np.float32)


def _slab(seed, n, box):
    """A membrane-shaped box: 40 % of the height holds zigzag chains of 12 beads in two leaflets (charges N(0, 0.3),
    neutral per chain), the rest waters on a jittered lattice; 0.1 charges per cubic Angstrom throughout.  Rows in the
    order chains, waters, then single neutralising pairs that fill up to n."""
    r = np.random.default_rng(seed)
    lx, ly, lz = box
    zc, half = 0.5 * lz, 0.2 * lz
    n_b = int(0.4 * n) // 12 * 12
    n_w = (n - n_b) // 3
    # chains: a lateral lattice per layer of chains, 12 beads along z, alternating sideways by the bond's rest
    layers = max(2, 2 * int(round(half / 20.0)))
    depth = 2.0 * half / layers
    chains = n_b // 12
    per = -(-chains // layers)
    mx = max(1, int(math.ceil(math.sqrt(per * lx / ly))))
    my = -(-per // mx)
    dz = depth / 12.0
    side = 0.5 * math.sqrt(max(0.0, 1.53 ** 2 - dz ** 2))
    c = np.arange(chains)
    lay, rest = c // per, c % per
    th = r.uniform(0.0, 2.0 * math.pi, layers)[lay]
    x0 = (rest % mx + 0.5) * lx / mx
    y0 = (rest // mx + 0.5) * ly / my
    k = np.arange(12)
    sgn = np.where(k % 2 == 0, 1.0, -1.0) * side
    bx = x0[:, None] + sgn * np.cos(th)[:, None]
    by = y0[:, None] + sgn * np.sin(th)[:, None]
    bz = (zc - half + lay * depth)[:, None] + (k + 0.5) * dz
    beads = np.stack([bx, by, bz], axis=2) + r.uniform(-0.15, 0.15, (chains, 12, 3))
    qb = r.normal(0.0, 0.3, (chains, 12))
    qb -= qb.mean(axis=1, keepdims=True)
    # waters: O sites of a lattice over the two outer layers
    hz = lz - 2.0 * half - 2.0
    a = (lx * ly * hz / max(1, n_w)) ** (1.0 / 3.0)
    m = np.maximum(1, np.floor(np.array([lx, ly, hz]) / a).astype(np.int64))
    while m.prod() < n_w:
        m[np.argmax(np.array([lx, ly, hz]) / m)] += 1
    site = r.permutation(int(m.prod()))[:n_w]
    step = np.array([lx, ly, hz]) / m
    o = (np.stack([site % m[0], site // m[0] % m[1], site // (m[0] * m[1])], axis=1) + 0.5) * step
    o += r.uniform(-0.25, 0.25, (n_w, 3))
    o[:, 2] += zc + half + 1.0
    rot = W.random_rotations(r, n_w)
    s, co = math.sin(W.THETA_HOH / 2) * W.R_OH, math.cos(W.THETA_HOH / 2) * W.R_OH
    local = np.array([[0.0, 0.0, 0.0], [s, 0.0, co], [-s, 0.0, co]])
    w = o[:, None, :] + np.einsum("nij,kj->nki", rot, local)
    rows = [np.concatenate([beads.reshape(-1, 3), qb.reshape(-1, 1)], axis=1),
            np.concatenate([w.reshape(-1, 3), np.tile([W.Q_O, W.Q_H, W.Q_H], n_w)[:, None]], axis=1)]
    left = n - n_b - 3 * n_w
    if left:        # up to two charges more, in the gap between the chains and the waters
        e = np.zeros((left, 4))
        e[:, 0], e[:, 1], e[:, 2] = (np.arange(left) + 0.5) * 0.4 * lx, 0.5 * ly, zc - half - 0.4
        e[:, 3] = 0.5 - np.arange(left) if left == 2 else 0.0
        rows.append(e)
    out = np.concatenate(rows)
    out[:, :3] = np.mod(out[:, :3], np.asarray(box))
    return out.astype(np.float32)


SYSTEMS = {"water": _water, "ions": _ions, "slab": _slab}


def _box(case):
    return (case["lx"], case["ly"], case["lz"])


def _grid(case):
    return (case["gx"], case["gy"], case["gz"])


def _kw(case):
    conv, points, ratio = FORMS[case["form"]]
    return dict(conv=conv, spread_points=points, spread_sigma_over_h=ratio, multilevel=case["multilevel"])


def _rows(case, seed):
    return SYSTEMS[case["system"]](1000 + seed, case["n"], _box(case))


def _stream_sizes(case):
    """Charges of each system of a batch: evenly spread over the logarithm of 2,000 to 60,000, in a mixed order."""
    k = case["n"]
    ns = [3 * int(2000.0 * 30.0 ** ((i + 0.5) / k) / 3.0) for i in range(k)]
    return [ns[(7 * i + 3) % k] if k % 7 else ns[i] for i in range(k)]


def _stream_grid(box):
    """The serving stream's grid rule: about 1 Angstrom, a multiple of 8, at least 24 points per axis."""
    g = max(24, int(round(box[0] / 8.0)) * 8)
    return (g, g, g)


def _stream(case, seed):
    """The batch's systems: (box, grid, r_c, rows) each."""
    res = []
    for i, n in enumerate(_stream_sizes(case)):
        box, rows = W.lattice_water_box((1000 + seed) * 1000 + i, n, DENSITY)
        res.append((box, _stream_grid(box), case["r_c"], rows))
    return res


def prepare(case, seed):
    if case["entry"] == "server":
        conv, points, ratio = FORMS[case["form"]]
        todo = []
        for box, grid, r_c, rows in _stream(case, seed):
            p = usr.make_params(box, grid, r_c, "C1_B2", max_atoms=rows.shape[0], conv=conv, spread_points=points,
                                spread_sigma_over_h=ratio)
            todo.append((p, torch.from_numpy(rows).pin_memory(), torch.empty(rows.shape, dtype=torch.float32,
                                                                             pin_memory=True)))
        return {"entry": "server", "server": usr.Server(hbm_budget_bytes=16 << 30, slots=8), "todo": todo}
    rows = torch.from_numpy(_rows(case, seed))
    n = rows.shape[0]
    ctx = usr.USeries(_box(case), _grid(case), case["r_c"], "C1_B2", max_atoms=n, **_kw(case))
    s = {"entry": case["entry"], "ctx": ctx, "n": n}
    if case["entry"] == "host":
        s["x"] = rows.pin_memory()
        s["out"] = torch.empty((n, 4), dtype=torch.float32, pin_memory=True)
        return s
    x = rows.cuda()
    if case["entry"] == "grad":
        s["xyz"] = x[:, :3].contiguous().requires_grad_(True)
        s["q"] = x[:, 3].contiguous().requires_grad_(True)
    else:
        s["x"] = x
        s["out"] = torch.empty((n, 4), dtype=torch.float32, device="cuda")
    return s


def run(state):
    entry = state["entry"]
    if entry == "server":
        server = state["server"]
        for p, x, out in state["todo"]:
            server.submit(p, x, out)
        server.wait()
        server.poll()
        return [t[2] for t in state["todo"]]
    ctx = state["ctx"]
    if entry == "grad":
        e = usr_energy(state["xyz"], state["q"], ctx)
        return list(torch.autograd.grad(e, (state["xyz"], state["q"])))
    call = usr.usr_eval_host if entry == "host" else usr.usr_eval
    call(ctx.ctx, state["n"], state["x"].data_ptr(), state["out"].data_ptr(), None)
    return state["out"]


# ---------------------------------------------------------------- work

def _pair_flops(n, box, r_c):
    """40 flops per unordered pair inside the cutoff (displacement, 1/r, the far function and its derivative, the
    force and the potential on both)."""
    return 40.0 * 0.5 * n * (4.0 / 3.0 * math.pi * r_c ** 3) * n / (box[0] * box[1] * box[2])


def _one_work(n, box, grid, r_c, kw):
    """Charges read once, forces and potentials written once; pair flops, the stencils (2 flops per point to spread,
    8 to gather value and gradient) and the per-axis convolutions of every far Gaussian."""
    info = usr.usr_plan(usr.make_params(box, grid, r_c, "C1_B2", max_atoms=n, **kw))
    g = float(grid[0] * grid[1] * grid[2])
    fine, coarse = info.n_terms - info.n_terms_coarse, info.n_terms_coarse
    conv = 2.0 * g * sum(grid) * (fine + coarse / 16.0)
    flops = _pair_flops(n, box, r_c) + 10.0 * kw["spread_points"] ** 3 * n + conv
    return 32.0 * n, flops


def work(case):
    if case["entry"] == "server":
        conv, points, ratio = FORMS[case["form"]]
        kw = dict(conv=conv, spread_points=points, spread_sigma_over_h=ratio)
        each = [_one_work(n, _cube(n), _stream_grid(_cube(n)), case["r_c"], kw) for n in _stream_sizes(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    b, f = _one_work(case["n"], _box(case), _grid(case), case["r_c"], _kw(case))
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- exact

_B, _R0, _W0 = 2.0, 1.98925368390802627, 0.994446492762232252     # Table 2, C1 construction at b = 2


def _terms(r_c):
    """(amplitude, width) of every Gaussian of the far function (Eqs. 23, 24)."""
    sigma = r_c / _R0
    c = 2.0 * math.log(_B) / math.sqrt(2.0 * math.pi * sigma * sigma)
    return [(c * (_W0 if j == 0 else _B ** -j), sigma * _B ** j) for j in range(67)]


def _exact(rows, box, r_c):
    """Forces and potentials (n, 4) in 64 bits: the direct pair sum of Eq. 20 over minimum images (every cutoff is
    at most a third of the box), the exact k-space sum of the far function (k = 0 dropped) and the self term."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x = torch.as_tensor(rows[:, :3], device=dev, dtype=torch.float64)
    q = torch.as_tensor(rows[:, 3], device=dev, dtype=torch.float64)
    L = torch.tensor(box, device=dev, dtype=torch.float64)
    n = x.shape[0]
    terms = _terms(r_c)
    phi = torch.zeros(n, device=dev, dtype=torch.float64)
    F = torch.zeros((n, 3), device=dev, dtype=torch.float64)
    step = max(1, min(n, 60_000_000 // n))
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        r2 = torch.zeros((i1 - i0, n), device=dev, dtype=torch.float64)
        for a in range(3):
            d = x[i0:i1, a, None] - x[None, :, a]
            d -= L[a] * torch.round(d / L[a])
            r2 += d * d
        r2[torch.arange(i1 - i0, device=dev), torch.arange(i0, i1, device=dev)] = 1e30
        i, j = torch.nonzero(r2 < r_c * r_c, as_tuple=True)
        u = r2[i, j]
        del r2, d
        r = torch.sqrt(u)
        far = torch.zeros_like(u)
        slope = torch.zeros_like(u)             # -dF/dr / r
        for amp, s in terms:
            g = amp * torch.exp(u * (-0.5 / (s * s)))
            far += g
            slope += g / (s * s)
        phi.index_add_(0, i + i0, q[j] * (1.0 / r - far))
        w = q[i + i0] * q[j] * (1.0 / (u * r) - slope)
        dv = x[i + i0] - x[j]
        dv -= L * torch.round(dv / L)
        F.index_add_(0, i + i0, w[:, None] * dv)
    # far: modes up to exp(-k^2 s_0^2 / 2) of 1e-17 of the first, half of them (S(-k) is the conjugate of S(k))
    s0 = terms[0][1]
    kmax = math.sqrt(2.0 * 39.0) / s0
    V = box[0] * box[1] * box[2]
    m = [int(kmax * b / (2.0 * math.pi)) for b in box]
    ph = [torch.exp(1j * (2.0 * math.pi / L[a]) * x[:, a, None] * torch.arange(-m[a], m[a] + 1, device=dev))
          for a in range(3)]
    kv = [2.0 * math.pi / box[a] * torch.arange(-m[a], m[a] + 1, device=dev, dtype=torch.float64) for a in range(3)]
    phi_far = torch.zeros(n, device=dev, dtype=torch.float64)
    grad = torch.zeros((n, 3), device=dev, dtype=torch.float64)
    for iz in range(m[2], 2 * m[2] + 1):        # k_z >= 0, weight 2 above the plane k_z = 0
        wt = 1.0 if iz == m[2] else 2.0
        kz = float(kv[2][iz])
        keep = int(math.sqrt(max(0.0, kmax * kmax - kz * kz)) * box[1] / (2.0 * math.pi)) + 1
        y0, y1 = max(0, m[1] - keep), min(2 * m[1] + 1, m[1] + keep + 1)
        k2 = kv[0][:, None] ** 2 + kv[1][None, y0:y1] ** 2 + kz * kz
        Fh = torch.zeros_like(k2)
        for amp, s in terms:
            Fh += amp * (2.0 * math.pi * s * s) ** 1.5 * torch.exp(-0.5 * s * s * k2)
        Fh[k2 == 0.0] = 0.0
        qz = q * ph[2][:, iz]
        ey = ph[1][:, y0:y1]
        S = ph[0].t() @ (qz[:, None] * ey)                                  # sum_i q_i exp(i k r_i)
        T = Fh * S.conj()
        U = ph[0] @ T                                                       # (n, ky)
        c = U * ey * ph[2][:, iz, None]
        phi_far += wt / V * c.real.sum(dim=1)
        grad[:, 1] -= wt / V * (c.imag @ kv[1][y0:y1])
        grad[:, 2] -= wt / V * kz * c.imag.sum(dim=1)
        Ux = ph[0] @ (kv[0][:, None] * T)
        grad[:, 0] -= wt / V * (Ux * ey * ph[2][:, iz, None]).imag.sum(dim=1)
    F -= q[:, None] * grad
    sigma = r_c / _R0
    F0 = 2.0 * math.log(_B) / math.sqrt(2.0 * math.pi * sigma * sigma) * (_W0 + 1.0 / (_B - 1.0))
    return torch.cat([F, (phi + phi_far - F0 * q)[:, None]], dim=1)


def exact(case, seed):
    """The outputs of `run` in 64 bits; None where the direct sums would take too long."""
    if case["entry"] == "server":
        return [_exact(rows, box, r_c) for box, _, r_c, rows in _stream(case, seed)]
    if case["n"] > 130000:
        return None
    out = _exact(_rows(case, seed), _box(case), case["r_c"])
    return [-out[:, :3], out[:, 3]] if case["entry"] == "grad" else out
