"""Cases that stand for what a user has this library do, timed through its public calls.

A time step is a few hundred roundings of sums of MPS (lincomb_round), a few
tens of products (hadamard_fit), and, now and then, the contraction of the
populations to rho and u; a simulation is set up by compressing its geometry
(from_dense).  Most cases are one such call on inputs shaped like a step's:
lattices of 8^3 to 256^3 cells, bonds of 8 to 128, one to nineteen jobs at a
time, FP64, FP32 and mixed precision; two are whole time steps.

An input MPS is a constant plus a sum of random tensor trains of decreasing
amplitude (1e-3 down to the rounding noise of its type), as the populations of a
weakly perturbed flow are: the singular values of every bond decay over the
whole range and fill the bond.  Results are compared as the fields they
represent (cores are fixed only up to a gauge), in the type they are stored in.
"""
import math

import numpy as np
import torch

from paper_2512_07615_gb300 import native, tnlbm

PRECISION = {"f64": native.FP64, "f32": native.FP32, "mixed": native.MIXED}
# largest work a drawn rounding may have: sites * bond^3 * jobs, by precision
ROUND_LIMIT = {"f64": 18 * 45 ** 3 * 3, "f32": 21 * 64 ** 3 * 9, "mixed": 21 * 64 ** 3 * 9}


def listed():
    return [
        # the smallest rounding: one sum on an 8^3 lattice, all latency
        dict(name="round_smallest", kind="round", precision="f32", n=3, bond=8, chi=8, jobs=1, terms="sum", eps=1e-7),
        # streaming towards the z walls of a 32^3 channel in FP64: one axis shift
        # and the bounce-back term of every moving population, untruncated
        dict(name="round_walls_f64", kind="round", precision="f64", n=5, bond=12, chi=16, jobs=18, terms="walls",
             eps=1e-10),
        # sums of 64^3 populations in FP64 at an odd bond cap
        dict(name="round_sum_f64_odd", kind="round", precision="f64", n=6, bond=45, chi=45, jobs=3, terms="sum",
             eps=1e-10),
        # the first level of the moment sums of a 128^3 step at bond 64, FP32
        dict(name="round_sum_f32", kind="round", precision="f32", n=7, bond=64, chi=64, jobs=9, terms="sum", eps=1e-7),
        # streaming of the 19 populations of a periodic 64^3 box at an odd bond, FP32
        dict(name="round_shift_f32_odd", kind="round", precision="f32", n=6, bond=37, chi=37, jobs=19, terms="shift",
             eps=1e-7),
        # the moment sums of the 128^3 step in mixed precision (the benchmark's mode)
        dict(name="round_sum_mixed", kind="round", precision="mixed", n=7, bond=64, chi=64, jobs=9, terms="sum",
             eps=1e-7),
        # sums of 256^3 populations at bond 128, mixed (the branching vessel's shapes)
        dict(name="round_wide_mixed", kind="round", precision="mixed", n=8, bond=128, chi=128, jobs=2, terms="sum",
             eps=1e-7),
        # the six products J_d u_e of a 128^3 step at bond 64: the variational fit, FP32
        dict(name="fit_f32", kind="fit", precision="f32", n=7, bond=64, bond_c=64, jobs=6),
        # set-up: a 64^3 sphere pack compressed to a mask MPS
        dict(name="mask_build", kind="mask", n=6, chi=48, radius=5.0, fraction=0.35),
        # output: rho and u of a 128^3 simulation at bond 64 on the host
        dict(name="fields_128", kind="fields", n=7, bond=64),
        # whole calls: a step from a checkpoint, then rho and u.  A 16^3 channel with
        # a box obstacle, z walls and a body force, FP64 with exact products
        dict(name="step_channel_f64", kind="step", precision="f64", n=4, chi=32, flow="channel", eps=1e-10),
        # a periodic 64^3 box of smooth waves, mixed precision
        dict(name="step_waves_mixed", kind="step", precision="mixed", n=6, chi=32, flow="waves", eps=1e-7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round", "round", "round", "round", "fit", "mask", "fields", "step"])
    if kind == "round":
        precision = rng.choice(["f64", "f32", "mixed"])
        n, jobs = rng.randint(3, 7), rng.randint(1, 19)
        bond = _log_int(rng, 6, 90)
        while 3 * n * bond ** 3 * jobs > ROUND_LIMIT[precision]:
            if jobs > 1:
                jobs -= 1
            else:
                bond -= 1
        chi = bond if rng.random() < 0.6 else min(2 * bond, 90 if precision != "f64" else 45)
        chi = max(chi, bond)
        return dict(kind="round", precision=precision, n=n, bond=bond, chi=chi, jobs=jobs,
                    terms=rng.choice(["sum", "shift", "walls"]), eps=1e-10 if precision == "f64" else 1e-7)
    if kind == "fit":
        return dict(kind="fit", precision="f32", n=rng.randint(4, 7), bond=_log_int(rng, 8, 64),
                    bond_c=_log_int(rng, 8, 64), jobs=rng.randint(1, 6))
    if kind == "mask":
        n = rng.randint(4, 6)
        return dict(kind="mask", n=n, chi=_log_int(rng, 8, 48), radius=round(rng.uniform(2.0, 6.0), 2),
                    fraction=round(rng.uniform(0.2, 0.4), 2))
    if kind == "fields":
        return dict(kind="fields", n=rng.randint(4, 7), bond=_log_int(rng, 8, 64))
    if rng.random() < 0.5:
        return dict(kind="step", precision="f64", n=rng.randint(3, 4), chi=rng.randint(28, 32), flow="channel", eps=1e-10)
    return dict(kind="step", precision="mixed", n=rng.randint(4, 6), chi=rng.randint(26, 32), flow="waves", eps=1e-7)


# ---------------------------------------------------------------- inputs
def _blocks(L, rho, count, gen):
    """count random tensor trains of L sites and bond rho with orthonormal rows
    (entries of order one): per site an array (count, r, 2, r')."""
    r = [min(rho, 2 ** k, 2 ** (L - k)) for k in range(L + 1)]
    out = []
    for k in range(L):
        g = torch.randn(count, 2 * r[k + 1], r[k], generator=gen, dtype=torch.float64)
        q = torch.linalg.qr(g)[0]
        out.append(math.sqrt(2.0) * q.transpose(1, 2).reshape(count, r[k], 2, r[k + 1]))
    return out


def _feasible_ends(cores):
    """The same tensor train with bonds of at most 2^k and 2^(L-k)."""
    cores, L = list(cores), len(cores)
    for k in range(L - 1):
        m = cores[k].reshape(-1, cores[k].shape[2])
        if 2 ** (k + 1) > m.shape[1]:
            break
        cores[k] = torch.eye(2 ** (k + 1), dtype=torch.float64).reshape(2 ** k, 2, 2 ** (k + 1))
        cores[k + 1] = torch.einsum("ab,bsc->asc", m, cores[k + 1])
    for k in range(L - 1, 0, -1):
        m = cores[k].reshape(cores[k].shape[0], -1)
        if 2 ** (L - k) > m.shape[0]:
            break
        cores[k] = torch.eye(2 ** (L - k), dtype=torch.float64).reshape(2 ** (L - k), 2, 2 ** (L - 1 - k))
        cores[k - 1] = torch.einsum("asb,bc->asc", cores[k - 1], m)
    return cores


def _field(L, bond, gen, const, amp, decades):
    """Cores of const + a sum of trains of bond four, amplitudes amp down to
    amp * 10^-decades, of total bond `bond`."""
    parts = [(1, [torch.ones(1, 1, 2, 1, dtype=torch.float64) for _ in range(L)])] if const else []
    rest = bond - len(parts)
    sizes = [4] * (rest // 4) + ([rest % 4] if rest % 4 else [])
    if rest // 4:
        parts.append((rest // 4, _blocks(L, 4, rest // 4, gen)))
    if rest % 4:
        parts.append((1, _blocks(L, rest % 4, 1, gen)))
    a = [amp * 10.0 ** (-decades * i / max(1, len(sizes) - 1)) for i in range(len(sizes))]
    weights = torch.tensor(([const] if const else []) + a, dtype=torch.float64)
    cores = []
    for k in range(L):
        mats = []
        at = 0
        for count, p in parts:
            c = p[k]
            if k == 0:
                c = c * weights[at:at + count].reshape(-1, 1, 1, 1)
            at += count
            r0, r1 = c.shape[1], c.shape[3]
            z = torch.zeros(count, r0, 2, count, r1, dtype=torch.float64)
            i = torch.arange(count)
            z[i, :, :, i, :] = c
            mats.append(z.reshape(count * r0, 2, count * r1))
        if k == 0:        # rows of the blocks share the one index of the left end
            mats = [m.sum(0, keepdim=True) for m in mats]
        if k == L - 1:
            mats = [m.sum(2, keepdim=True) for m in mats]
        r0, r1 = [sum(m.shape[0] for m in mats), sum(m.shape[2] for m in mats)]
        if k == 0:
            c = torch.cat(mats, 2)
        elif k == L - 1:
            c = torch.cat(mats, 0)
        else:
            c = torch.zeros(r0, 2, r1, dtype=torch.float64)
            i = j = 0
            for m in mats:
                c[i:i + m.shape[0], :, j:j + m.shape[2]] = m
                i, j = i + m.shape[0], j + m.shape[2]
        cores.append(c)
    return _feasible_ends(cores)


def _device(cores, cap, precision):
    X = tnlbm.DeviceMps(len(cores), cap, precision)
    flat = torch.zeros(X.data.numel(), dtype=torch.float64)
    for k, c in enumerate(cores):
        o = tnlbm.mps_offset(X.L, cap, k)
        flat[o:o + c.numel()] = c.reshape(-1)
    X.data.copy_(flat.to(X.data.dtype))
    X.ranks.copy_(torch.tensor([1] + [c.shape[2] for c in cores], dtype=torch.int32))
    return X


def _gen(seed, salt=0):
    return torch.Generator().manual_seed(1000003 * int(seed) + salt)


def _decades(precision):
    return 8.0 if precision == "f64" else 5.0


def _round_operands(case, seed):
    """Per job the two operands' cores."""
    L, gen = 3 * case["n"], _gen(seed)
    return [[_field(L, case["bond"], gen, w, 1e-3 * w, _decades(case["precision"])) for w in (1.0 / 18.0, 1.0 / 36.0)]
            for _ in range(case["jobs"])]


def _plane(L, axis, high):
    """The indicator of x_axis = 0 (or N - 1) as per-site pairs."""
    v = np.ones((L, 2))
    for k in range(axis, L, 3):
        v[k] = (0.0, 1.0) if high else (1.0, 0.0)
    return v


def _fit_operands(case, seed):
    """Per job a momentum-like factor and a factor 1 + 2e-6 (fluctuations), the
    inverse density of a weakly compressible flow."""
    L, gen = 3 * case["n"], _gen(seed, 1)
    return [(_field(L, case["bond"], gen, 0.0, 1.0, 5.0), _field(L, case["bond_c"], gen, 1.0, 2e-6, 2.0))
            for _ in range(case["jobs"])]


def _spheres(case, seed):
    """Voxels of a periodic pack of overlapping spheres, on the GPU."""
    N, gen = 1 << case["n"], _gen(seed, 2)
    volume = 4.0 / 3.0 * math.pi * case["radius"] ** 3
    count = max(1, int(round(-math.log(1.0 - case["fraction"]) * N ** 3 / volume)))
    centres = (N * torch.rand(count, 3, generator=gen, dtype=torch.float64)).cuda()
    ax = torch.arange(N, dtype=torch.float64, device="cuda") + 0.5
    solid = torch.zeros((N, N, N), dtype=torch.bool, device="cuda")
    for c in centres:
        d = (ax[None, :] - c[:, None]).abs()
        d = torch.minimum(d, N - d).square()
        solid |= (d[0][:, None, None] + d[1][None, :, None] + d[2][None, None, :]) <= case["radius"] ** 2
    return solid.double()


def _modes(seed, count=12, kmax=2, amp=1e-3):
    """Plane waves (kx ky kz phase a_rho a_ux a_uy a_uz) of a smooth start."""
    r = np.random.default_rng(int(seed))
    rows = []
    for _ in range(count):
        k = np.zeros(3, dtype=int)
        while not k.any():
            k = r.integers(-kmax, kmax + 1, 3)
        rows.append([*k, r.uniform(0, 2 * math.pi), *r.uniform(-amp, amp, 4)])
    return np.array(rows)


def _box(case, seed):
    """A solid box inside the channel (corners on eighths of the axis, so that
    the step's bonds stay below the cap) and the body force."""
    N = 1 << case["n"]
    r = np.random.default_rng(int(seed))
    lo = N // 8 * r.integers(1, 4, 3)
    hi = N // 8 * r.integers(4, 8, 3)
    m = np.zeros((N, N, N), dtype=np.uint8)
    m[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] = 1
    return m, float(r.uniform(1e-6, 1e-5))


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "round":
        p, L = PRECISION[case["precision"]], 3 * case["n"]
        jobs = []
        keep = []
        for j, (X, Y) in enumerate(_round_operands(case, seed)):
            x, y = _device(X, case["bond"], p), _device(Y, case["bond"], p)
            keep += [x, y]
            if case["terms"] == "sum":
                jobs.append([tnlbm.plain(x), tnlbm.plain(y, -0.43)])
            elif case["terms"] == "shift":
                jobs.append([tnlbm.shift(x, j % 3, 1 if j % 2 else -1)])
            else:
                high = bool(j % 2)
                jobs.append([tnlbm.shift(x, 2, 1 if high else -1, cyclic=False), tnlbm.mask1(y, _plane(L, 2, high))])
        s["jobs_"] = jobs
        s["dst"] = [tnlbm.DeviceMps(L, case["chi"], p) for _ in jobs]
    elif kind == "fit":
        p, L = PRECISION[case["precision"]], 3 * case["n"]
        ops = _fit_operands(case, seed)
        s["B"] = [_device(b, case["bond"], p) for b, _ in ops]
        s["C"] = [_device(c, case["bond_c"], p) for _, c in ops]
        s["A"] = [tnlbm.DeviceMps(L, case["bond"], p) for _ in ops]
    elif kind == "mask":
        s["solid"] = _spheres(case, seed)
    elif kind == "fields":
        s["sim"] = tnlbm.Sim(case["n"], tau=0.7, chi_max=case["bond"], eps=1e-7, precision=native.MIXED,
                             force=(1e-5, 0.0, 0.0))
        s["sim"].set_populations([[c.numpy() for c in f] for f in _populations(case, seed)])
    elif case["flow"] == "channel":
        solid, force = _box(case, seed)
        s["sim"] = tnlbm.Sim(case["n"], tau=0.8, periodic=(1, 1, 0), solid=solid, chi_mask=16, force=(force, 0.0, 0.0),
                             chi_max=case["chi"], eps=case["eps"], precision=PRECISION[case["precision"]],
                             hadamard=native.HADAMARD_EXACT)
        s["start"] = s["sim"].get_populations()
    else:
        s["sim"] = tnlbm.Sim(case["n"], tau=0.7, modes=_modes(seed), force=(1e-5, 0.0, 0.0), chi_max=case["chi"],
                             eps=case["eps"], precision=PRECISION[case["precision"]])
        s["start"] = s["sim"].get_populations()
    return s


def run(s):
    kind = s["kind"]
    if kind == "round":
        tnlbm.lincomb_round(s["jobs_"], s["dst"], s["chi"], s["eps"])
        return [tnlbm.to_dense(d) for d in s["dst"]]
    if kind == "fit":
        tnlbm.hadamard_fit(s["B"], s["C"], s["A"], sweeps=2)
        return [tnlbm.to_dense(a) for a in s["A"]]
    if kind == "mask":
        return tnlbm.to_dense(tnlbm.from_dense(s["solid"], s["chi"], s["chi"], 1e-8))
    if kind == "fields":
        return s["sim"].macroscopic()
    # a step resumed from stored populations; rho and u as one array of the
    # simulation's own type
    s["sim"].set_populations(s["start"])
    s["sim"].step(1)
    rho, u = s["sim"].macroscopic()
    out = np.concatenate([rho[None], u])
    return out if s["precision"] == "f64" else out.astype(np.float32)


def _populations(case, seed):
    gen = _gen(seed, 3)
    w = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
    return [_field(3 * case["n"], case["bond"], gen, wi, 1e-3 * wi, 5.0) for wi in w]


# ---------------------------------------------------------------- work
def _bonds(L, r):
    return [min(r, 2 ** k, 2 ** (L - k)) for k in range(L + 1)]


def _elems(r):
    return sum(r[k] * 2 * r[k + 1] for k in range(len(r) - 1))


def _round_flops(L, wide, out):
    """QR of the wide cores and a truncated SVD of every centre matrix."""
    f = 0.0
    q = [min(wide[k], 2 ** k, 2 ** (L - k)) for k in range(L + 1)]
    for k in range(L):
        m, n = 2 * q[k], q[k + 1]
        f += 2.0 * q[k] * wide[k] * 2 * wide[k + 1] + 4.0 * m * n * n - 4.0 / 3.0 * n ** 3
        m, n = q[k], 2 * out[k + 1]
        lo, hi = min(m, n), max(m, n)
        f += 4.0 * hi * lo * lo + 8.0 * lo ** 3 + 2.0 * 2 * q[k] * q[k + 1] * out[k + 1]
    return f


def work(case):
    n = case["n"]
    L, cells = 3 * n, 8 ** n
    size = 8 if case.get("precision") == "f64" else 4
    if case["kind"] == "round":
        r, o = _bonds(L, case["bond"]), _bonds(L, min(case["chi"], 2 * case["bond"]))
        wide = [1 if k in (0, L) else (1 if case["terms"] == "sum" else 2) * r[k] + (0 if case["terms"] == "shift" else r[k])
                for k in range(L + 1)]
        terms = 1 if case["terms"] == "shift" else 2
        return dict(bytes=case["jobs"] * size * (terms * _elems(r) + cells),
                    flops=case["jobs"] * (_round_flops(L, wide, o) + 2.0 * cells * o[L // 2]))
    if case["kind"] == "fit":
        a, c = _bonds(L, case["bond"]), _bonds(L, case["bond_c"])
        site = [2.0 * (a[k] * c[k] * a[k] * 2 * a[k + 1] + a[k] * 2 * c[k] * c[k + 1] * a[k + 1] +
                       2 * a[k] * a[k + 1] * c[k + 1] * a[k + 1] + a[k + 1] * c[k + 1] * a[k + 1] * 2 * a[k])
                for k in range(L)]
        return dict(bytes=case["jobs"] * size * (_elems(a) + _elems(c) + cells),
                    flops=case["jobs"] * (5.0 * sum(site) + 2.0 * cells * a[L // 2]))
    if case["kind"] == "mask":
        r = _bonds(L, case["chi"])
        return dict(bytes=16 * cells, flops=sum(2.0 * (2 * r[k]) * (2 * r[k] + r[k + 1]) * (cells >> (k + 1))
                                                for k in range(L)) + 2.0 * cells * r[L // 2])
    if case["kind"] == "fields":
        r = _bonds(L, case["bond"])
        return dict(bytes=19 * 4 * _elems(r) + 4 * 8 * cells, flops=19 * 2.0 * cells * r[L // 2])
    # a step: its input and output populations; about 200 roundings and 10
    # products of bonds that such flows reach in one step (half the cap)
    r = _bonds(L, case["chi"] // 2)
    jobs = 250 if case["flow"] == "channel" else 180
    return dict(bytes=2 * 19 * size * _elems(r) + 4 * size * cells,
                flops=jobs * _round_flops(L, [1 if k in (0, L) else 2 * x for k, x in enumerate(r)], r))


# ---------------------------------------------------------------- the same in 64 bits
def _cells_order(n):
    """For every cell [x][y][z] the index of its site-ordered (bits interleaved) entry."""
    a = torch.arange(1 << n, device="cuda")
    spread = torch.zeros_like(a)
    for b in range(n):
        spread += ((a >> b) & 1) << (3 * b)
    return (spread[:, None, None] << 2) + (spread[None, :, None] << 1) + spread[None, None, :]


def _dense(cores, dtype):
    """The field of the cores as stored in dtype, in 64 bits."""
    cores = [c.to(dtype).double().cuda() for c in cores]
    L = len(cores)
    left = cores[0].reshape(2, -1)
    for c in cores[1:L // 2]:
        left = (left @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    right = cores[-1].reshape(-1, 2)
    for c in reversed(cores[L // 2:-1]):
        right = (c.reshape(-1, c.shape[2]) @ right).reshape(c.shape[0], -1)
    return (left @ right).reshape(-1)[_cells_order(L // 3)]


def _shifted(x, axis, offset, cyclic):
    """x(cell + offset along axis), zero beyond the domain if not cyclic."""
    y = torch.roll(x, -offset, axis)
    if not cyclic:
        y = y.clone()
        y.narrow(axis, x.shape[axis] - 1 if offset > 0 else 0, 1).zero_()
    return y


def _exact_mask(case, seed):
    """TT-SVD of the voxels by eigenvectors of the unfoldings' Gram matrices."""
    n, L = case["n"], 3 * case["n"]
    v = _spheres(case, seed)
    order = _cells_order(n)
    m = torch.empty(8 ** n, dtype=torch.float64, device="cuda")
    m[order.reshape(-1)] = v.reshape(-1)
    delta2 = (1e-8 * float(m.norm())) ** 2 / (L - 1)
    cores, r = [], 1
    for _ in range(L - 1):
        m = m.reshape(2 * r, -1)
        lam, vec = torch.linalg.eigh(m @ m.T)
        lam, vec = lam.flip(0).clamp(min=0.0), vec.flip(1)
        floor = 1e-12 * float(lam[0])
        cap = min(case["chi"], *m.shape)
        tails = torch.cat([lam.flip(0).cumsum(0).flip(0), lam.new_zeros(1)]).cpu()
        keep = next((q for q in range(1, cap + 1) if tails[q] <= max(delta2, floor)), cap)
        u = vec[:, :keep].contiguous()
        cores.append(u.reshape(r, 2, keep).cpu())
        m, r = u.T @ m, keep
    cores.append(m.reshape(r, 2, 1).cpu())
    return _dense(cores, torch.float64)


_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
      (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _velocity(f, force, fluid):
    rho = f.sum(0)
    j = torch.stack([sum(c[d] * f[i] for i, c in enumerate(_C) if c[d]) for d in range(3)])
    j = j + 0.5 * torch.tensor(force, dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1) * fluid
    return rho, torch.where(rho > 0.5, j / torch.where(rho > 0.5, rho, 1.0), 0.0)


def _exact_step(case, seed):
    """One full-grid BGK step (D3Q19) with 1/rho to second order about its mean."""
    N = 1 << case["n"]
    ax = torch.arange(N, dtype=torch.float64, device="cuda")
    fluid = torch.ones(N, N, N, dtype=torch.float64, device="cuda")
    if case["flow"] == "channel":
        solid, F = _box(case, seed)
        fluid -= torch.from_numpy(solid).cuda()
        force, tau, periodic = (F, 0.0, 0.0), 0.8, (1, 1, 0)
        f = torch.stack([w * fluid for w in _W])
    else:
        force, tau, periodic = (1e-5, 0.0, 0.0), 0.7, (1, 1, 1)
        f = torch.stack([w * fluid for w in _W])
        for kx, ky, kz, phase, a_rho, *a_u in _modes(seed):
            wave = torch.cos(2 * math.pi / N * (kx * ax[:, None, None] + ky * ax[None, :, None] + kz * ax[None, None, :])
                             + phase)
            for i, c in enumerate(_C):
                f[i] += _W[i] * (a_rho + 3.0 * sum(c[d] * a_u[d] for d in range(3))) * wave
    rho = f.sum(0)
    rho0 = rho.sum() / fluid.sum()
    drho = rho - rho0
    inv = 1 / rho0 - drho / rho0 ** 2 + drho ** 2 / rho0 ** 3
    J = [sum(c[d] * f[i] for i, c in enumerate(_C) if c[d]) + tau * force[d] * fluid for d in range(3)]
    u = [x * inv for x in J]
    post = []
    for i, c in enumerate(_C):
        e = rho - 1.5 * sum(J[d] * u[d] for d in range(3))
        e = e + 3.0 * sum(c[d] * J[d] for d in range(3))
        for d in range(3):
            for q in range(d, 3):
                e = e + (4.5 if d == q else 9.0) * c[d] * c[q] * J[d] * u[q]
        post.append((1 - 1 / tau) * f[i] + _W[i] / tau * e)

    def stream(x, c):
        for d in range(3):
            if c[d]:
                x = _shifted(x, d, -c[d], bool(periodic[d]))
        return x

    back = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
    new = []
    for i, c in enumerate(_C):
        x = stream(post[i], c)
        if c[2] and not periodic[2]:
            at = 0 if c[2] > 0 else N - 1
            x[:, :, at] += post[back[i]][:, :, at]
        new.append(x)
    if case["flow"] == "channel":
        g = [x * (1 - fluid) for x in new]
        new = [new[0]] + [new[i] - g[i] + stream(g[back[i]], _C[i]) for i in range(1, 19)]
    rho, v = _velocity(torch.stack(new), force, fluid)
    return torch.cat([rho[None], v])


def exact(case, seed):
    kind = case["kind"]
    if kind == "round":
        dtype = torch.float64 if case["precision"] == "f64" else torch.float32
        out = []
        for j, (X, Y) in enumerate(_round_operands(case, seed)):
            x = _dense(X, dtype)
            if case["terms"] == "sum":
                out.append(x - 0.43 * _dense(Y, dtype))
            elif case["terms"] == "shift":
                out.append(_shifted(x, j % 3, 1 if j % 2 else -1, True))
            else:
                high = bool(j % 2)
                x = _shifted(x, 2, 1 if high else -1, False)
                at = -1 if high else 0
                x[:, :, at] += _dense(Y, dtype)[:, :, at]
                out.append(x)
        return out
    if kind == "fit":
        return [_dense(b, torch.float32) * _dense(c, torch.float32) for b, c in _fit_operands(case, seed)]
    if kind == "mask":
        return _exact_mask(case, seed)
    if kind == "fields":
        f = torch.stack([_dense(p, torch.float32) for p in _populations(case, seed)])
        return _velocity(f, (1e-5, 0.0, 0.0), 1.0)
    return _exact_step(case, seed).cpu().numpy()
