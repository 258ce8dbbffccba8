"""Measured workloads of the tree builder, each through the calls a program makes.

    build    tb.build + tb.moments rebuilding a kept tree in place: the step of
             an N-body program.  With "fixed" the build is given a cell
             capacity and never waits for the GPU; without, it reads the cell
             count back and sizes the arrays itself (they have room already).
    batched  tb.build_batched: one tree per particle set (halo catalogues,
             zoom regions, independent subvolumes).
    walk     tb.walk on a built tree: accelerations of every particle.
    reorder  tb.reorder of a program's positions, velocities, masses and ids
             into key order, done every few steps.
    noalloc  tb.keys_sorted_noalloc: keys and stable sort without allocation.

Particles are drawn on the GPU: uniform boxes, Plummer spheres, exponential
discs, NFW haloes on a uniform background ("clustered"), and that mix moved
to [1000, 1001)^3 with log-normal masses ("stress").
"""
import math

import torch

import paper_2312_06102_gb300 as tb

F64 = torch.float64
DEV = "cuda"


# ------------------------------------------------------------------ cases

def _build(name, n, dist, n_crit=16, mode="comp", key="morton", fixed=True, sorted_pos=False,
           pow2=False, mass=True, skip=0, pair=False):
    return dict(name=name, kind="build", n=n, dist=dist, n_crit=n_crit, mode=mode, key=key,
                fixed=fixed, sorted_pos=sorted_pos, pow2=pow2, mass=mass, skip=skip, pair=pair)


def listed():
    return [
        # a small system stepped many times: launches and latency are the cost
        _build("build_3k", 3001, "uniform", n_crit=10),
        # the plain single build of 65,536 uniform particles
        _build("build_64k", 65536, "uniform"),
        # an ordinary system, the cell count read back at each build, one species
        # of a shared position array (not 16-byte aligned), default masses, the
        # centres of mass taken as com + com_lo
        _build("build_1m_exact", 1000003, "plummer", n_crit=8, fixed=False, mass=False, skip=1,
               pair=True),
        # disc galaxy with Hilbert keys, sorted particles kept, power-of-two root
        _build("build_4m_hilbert", 4194304, "disk", key="hilbert", sorted_pos=True, pow2=True),
        # log-normal masses far from the origin, FP64 moments
        _build("build_6m_fp64", 6000000, "stress", mode="fp64"),
        # Plummer sphere, deep levels in the core
        _build("build_16m", 16777216, "plummer"),
        # the largest configured build: 2^27 clustered particles
        _build("build_128m", 134217728, "clustered"),
        # a halo catalogue: a few hundred small sets
        dict(name="batched_300", kind="batched", sets=300, nmin=64, nmax=4096, n_crit=10),
        # the configured batch: 4,096 sets of 256 to 65,536 particles
        dict(name="batched_4096", kind="batched", sets=4096, nmin=256, nmax=65536, n_crit=16),
        # forces of a million particles at the usual opening angle
        dict(name="walk_1m", kind="walk", n=1048576, dist="plummer", n_crit=10, theta=0.75,
             group=128, quad=True),
        # a program's particle arrays put into key order
        dict(name="reorder_16m", kind="reorder", n=16777213, dist="clustered"),
        # keys and order of a sub-sample inside another component's loop
        dict(name="noalloc_300k", kind="noalloc", n=300007, dist="clustered"),
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, n))


def draw(rng):
    dist = rng.choice(["uniform", "plummer", "disk", "clustered", "stress"])
    kind = rng.choice(["build", "build", "build", "build", "batched", "walk", "reorder", "noalloc"])
    if kind == "build":
        return dict(kind="build", n=_log_int(rng, 1000, 1 << 26), dist=dist,
                    n_crit=rng.choice([8, 10, 16, 16, 32, 64]),
                    mode=rng.choice(["comp", "comp", "comp", "plain", "fp64"]),
                    key=rng.choice(["morton", "morton", "morton", "hilbert"]),
                    fixed=rng.random() < 0.75, sorted_pos=rng.random() < 0.25,
                    pow2=rng.random() < 0.25, mass=rng.random() < 0.75,
                    skip=rng.choice([0, 0, 0, 1]), pair=rng.random() < 0.25)
    if kind == "batched":
        nmin = _log_int(rng, 32, 1024)
        nmax = _log_int(rng, 2 * nmin, 65536)
        return dict(kind="batched", sets=_log_int(rng, 16, 4096), nmin=nmin, nmax=nmax,
                    n_crit=rng.choice([8, 10, 16, 32]))
    if kind == "walk":
        return dict(kind="walk", n=_log_int(rng, 2000, 1 << 21),
                    dist=rng.choice(["plummer", "disk", "clustered"]),
                    n_crit=rng.choice([8, 10, 16]), theta=rng.choice([0.5, 0.75, 1.0]),
                    group=rng.choice([32, 64, 128, 256]), quad=rng.random() < 0.75)
    if kind == "reorder":
        return dict(kind="reorder", n=_log_int(rng, 1000, 1 << 25), dist=dist)
    return dict(kind="noalloc", n=_log_int(rng, 1000, tb.NOALLOC_MAX_N), dist=dist)


# ----------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _directions(g, n):
    mu = 2.0 * _rand(g, n) - 1.0
    phi = 2.0 * math.pi * _rand(g, n)
    s = (1.0 - mu * mu).clamp_(min=0.0).sqrt_()
    return torch.stack([s * phi.cos(), s * phi.sin(), mu], dim=1)


def _plummer(g, n, a):
    """Radii of a Plummer sphere of scale radius a, truncated at 20 a."""
    u = _rand(g, n) * (400.0 / 401.0) ** 1.5
    r = a / (u.clamp_(min=1e-300).pow_(-2.0 / 3.0) - 1.0).sqrt_()
    return 0.5 + r[:, None] * _directions(g, n)


def _nfw(g, n, c):
    """NFW radii in units of the scale radius: enclosed mass inverted from a table."""
    x = c * torch.linspace(0.0, 1.0, 65537, device=DEV, dtype=F64) ** 2
    m = torch.log1p(x) - x / (1.0 + x)
    t = _rand(g, n) * m[-1]
    i = torch.searchsorted(m, t).clamp_(1, m.numel() - 1)
    w = (t - m[i - 1]) / (m[i] - m[i - 1])
    return x[i - 1] + w * (x[i] - x[i - 1])


def _clustered(g, n):
    """70% in NFW haloes with dN/dM ~ M^-1.9 (counts 100 to 10^6, rescaled to
    the total), 30% uniform; shuffled, in [0,1)^3."""
    nh = int(round(0.7 * n))
    halos = max(1, min(10000, nh // 100))
    u = _rand(g, halos)
    raw = (100.0 ** -0.9 + u * (1e6 ** -0.9 - 100.0 ** -0.9)) ** (1.0 / -0.9)
    cum = torch.cumsum(raw, 0)
    edge = torch.round(cum * (nh / cum[-1])).to(torch.int64)
    counts = torch.diff(edge, prepend=edge.new_zeros(1))
    r_s = (3.0 * counts / (4.0 * math.pi * 200.0 * n)) ** (1.0 / 3.0) / 10.0
    which = torch.repeat_interleave(torch.arange(halos, device=DEV), counts, output_size=nh)
    pos = _rand(g, halos, 3)[which]
    pos += (r_s[which] * _nfw(g, nh, 10.0))[:, None] * _directions(g, nh)
    pos -= pos.floor()
    pos = torch.cat([pos, _rand(g, n - nh, 3)])
    return pos[torch.randperm(n, generator=g, device=DEV)]


def _particles(g, n, dist):
    """Positions [n, 3] and masses [n], FP32."""
    mass = torch.full((n,), 1.0 / n, device=DEV, dtype=torch.float32)
    if dist == "uniform":
        pos = _rand(g, n, 3)
    elif dist == "plummer":
        pos = _plummer(g, n, 0.05)
    elif dist == "disk":
        # R ~ Gamma(2, 1): the sum of two exponentials; sech^2 heights
        r = 0.05 * (-(1.0 - _rand(g, n)).log_() - (1.0 - _rand(g, n)).log_()).clamp_(max=10.0)
        phi = 2.0 * math.pi * _rand(g, n)
        z = 0.005 * torch.atanh((2.0 * _rand(g, n) - 1.0).clamp_(-1.0 + 1e-8, 1.0 - 1e-8))
        pos = 0.5 + torch.stack([r * phi.cos(), r * phi.sin(), z], dim=1)
    else:
        pos = _clustered(g, n)
        if dist == "stress":
            pos += 1000.0
            z = torch.randn(n, generator=g, device=DEV, dtype=F64)
            mass = ((1.0 / n) * (2.0 * z).exp()).to(torch.float32)
    return pos.to(torch.float32), mass


def _inputs(case, seed):
    """(positions, masses or None, set offsets or None) of a case."""
    g = _gen(seed)
    if case["kind"] == "batched":
        # log-uniform sizes in an order of the seed's
        lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
        at = (torch.randperm(case["sets"], generator=g, device=DEV) + 0.5) / case["sets"]
        size = (lo + (hi - lo) * at.to(F64)).exp().floor().to(torch.int64)
        off = torch.zeros(case["sets"] + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(size, 0, out=off[1:])
        a = (math.log(0.01) + (math.log(0.2) - math.log(0.01)) * _rand(g, case["sets"])).exp()
        total = int(off[-1])
        which = torch.repeat_interleave(torch.arange(case["sets"], device=DEV), size, output_size=total)
        pos = _plummer(g, total, a[which]).to(torch.float32)
        return pos, (1.0 / size.to(F64)).to(torch.float32)[which], off
    skip = case.get("skip", 0)
    pos, mass = _particles(g, case["n"] + skip, case["dist"])
    if skip:
        pos, mass = pos[skip:], mass[skip:]
    return pos, mass if case.get("mass", True) else None, None


MODES = {"comp": tb.MOM_FP32_COMP, "plain": tb.MOM_FP32_PLAIN, "fp64": tb.MOM_FP64}


def _options(case):
    return dict(n_crit=case["n_crit"], mom_mode=MODES[case["mode"]], reorder=case["sorted_pos"],
                key_order=tb.KEYS_HILBERT if case["key"] == "hilbert" else tb.KEYS_MORTON,
                root_pow2=case["pow2"])


def _u64(t):
    return t.view(torch.int64)


def _capacity(case, n):
    """Room for the cells of any such input: 1.5 times the 4 n / n_crit of the
    clustered set, and what many small sets need."""
    return 6 * n // case["n_crit"] + 64 * case.get("sets", 16)


class _Array:
    """A device array of a tree, at its whole length; keeps the tree alive."""

    def __init__(self, tree, ptr, shape, typestr):
        self.tree = tree
        self.__cuda_array_interface__ = dict(shape=shape, typestr=typestr, data=(ptr, False),
                                             version=3, strides=None, stream=None)


def _arrays(t, n, cap, fp64=False, sets=0, sorted_pos=False, pair=False):
    """The tree's arrays at the lengths they have for every step of a program
    that keeps room for `cap` cells: [0, n_cells) and [0, n_leaves) are the
    tree, the rest is cleared once and never written."""
    u8, i32, i64, f32, f64 = "|u1", "<i4", "<i8", "<f4", "<f8"
    shapes = dict(pkey=((n,), i64), perm=((n,), i32), ckey=((cap,), i64), level=((cap,), u8),
                  parent=((cap,), i32), child_first=((cap,), i32), child_end=((cap,), i32),
                  pfirst=((cap,), i32), pend=((cap,), i32), leaf_cell=((n,), i32),
                  mass=((cap,), f32), com=((cap, 3), f32), quad=((cap, 6), f32),
                  aabb=((cap, 6), f32))
    if pair:
        shapes["com_lo"] = ((cap, 3), f32)
    if fp64:
        shapes.update(mass64=((cap,), f64), com64=((cap, 3), f64), quad64=((cap, 6), f64))
    if sorted_pos:
        shapes["pos_sorted"] = ((n, 4), f32)
    if sets:
        shapes.update(set_cell_offset=((sets + 1,), i64), set_root=((sets, 4), f64))
    out = {k: torch.as_tensor(_Array(t, getattr(t.c, k), *v), device=DEV) for k, v in shapes.items()}
    for v in out.values():
        v.zero_()
    return out


def _outputs(views):
    """com_lo means nothing by itself (com rounds either way): a program that
    wants it forms the centre com + com_lo in 64 bits."""
    if "com_lo" not in views:
        return views
    out = dict(views)
    out["centre"] = out["com"].double().add_(out.pop("com_lo"))
    return out


def _ready(t):
    status = t.sync()
    if status != 0:
        raise tb.TbError(status, "build")


def prepare(case, seed):
    pos, mass, off = _inputs(case, seed)
    st = dict(case=case, pos=pos, mass=mass, off=off)
    kind = case["kind"]
    if kind == "build":
        st["opt"] = _options(case)
        st["cap"] = cap = _capacity(case, case["n"])
        st["tree"] = t = tb.build(pos, mass, cell_capacity=cap, **st["opt"])
        _ready(t)
        st["views"] = _arrays(t, case["n"], cap, fp64=case["mode"] == "fp64",
                              sorted_pos=case["sorted_pos"], pair=case["pair"])
    elif kind == "batched":
        n = pos.shape[0]
        st["cap"] = cap = _capacity(case, n)
        st["tree"] = t = tb.build_batched(pos, mass, off, n_crit=case["n_crit"], cell_capacity=cap)
        _ready(t)
        st["views"] = _arrays(t, n, cap, sets=case["sets"])
    elif kind == "walk":
        st["tree"] = t = tb.build(pos, mass, n_crit=case["n_crit"])
        tb.moments(t, pos, mass)
        st["eps"] = 1e-3 * t.side
        st["acc"] = torch.empty_like(pos)
    elif kind == "reorder":
        st["tree"] = tb.build(pos, mass)
        g = _gen(seed + 1)
        n = case["n"]
        vel = torch.randn(n, 3, generator=g, device=DEV)
        ids = torch.arange(n, device=DEV)
        st["src"] = dict(pos=pos, vel=vel, mass=mass, ids=ids)
        st["dst"] = {k: torch.empty_like(v) for k, v in st["src"].items()}
    else:
        st["pkey"] = torch.empty(case["n"], dtype=torch.uint64, device=DEV)
        st["perm"] = torch.empty(case["n"], dtype=torch.int32, device=DEV)
    return st


# -------------------------------------------------------------------- run

def run(st):
    kind = st["case"]["kind"]
    if kind == "build":
        cap = st["cap"] if st["case"]["fixed"] else 0
        tb.build(st["pos"], st["mass"], cell_capacity=cap, tree=st["tree"], **st["opt"])
        tb.moments(st["tree"], st["pos"], st["mass"])
        return _outputs(st["views"])
    if kind == "batched":
        tb.build_batched(st["pos"], st["mass"], st["off"], n_crit=st["case"]["n_crit"],
                         cell_capacity=st["cap"], tree=st["tree"])
        return st["views"]
    if kind == "walk":
        c = st["case"]
        return tb.walk(st["tree"], c["theta"], st["eps"], n_group=c["group"], use_quad=c["quad"],
                       out=st["acc"])
    if kind == "reorder":
        for k, v in st["src"].items():
            tb.reorder(st["tree"], v, out=st["dst"][k])
        return st["dst"]
    status, root = tb.keys_sorted_noalloc(st["pos"], st["pkey"], st["perm"])
    if status != 0:
        raise tb.TbError(status, "tb_keys_sorted_noalloc")
    return dict(pkey=_u64(st["pkey"]), perm=st["perm"], root=root)


# ------------------------------------------------------------------- work

def work(case):
    """Each input read once, each output written once.  Cells: about 4 n /
    n_crit of them (0.43 n, 0.27 n and 0.11 n measured at n_crit 8, 16 and 32
    on the clustered set), 105 bytes each (29 of structure, 76 of moments)."""
    kind = case["kind"]
    if kind == "batched":
        r = math.log(case["nmax"] / case["nmin"])
        n = case["sets"] * (case["nmax"] - case["nmin"]) / r
        return dict(bytes=(16 + 12) * n + 105 * 4.0 * n / case["n_crit"], flops=60.0 * n)
    n = case["n"]
    if kind == "build":
        per_cell = 105 + (80 if case["mode"] == "fp64" else 0)
        per_n = 12 + (4 if case["mass"] else 0) + 12 + (16 if case["sorted_pos"] else 0)
        return dict(bytes=per_n * n + per_cell * 4.0 * n / case["n_crit"], flops=60.0 * n)
    if kind == "walk":
        # 1,200 interactions a particle measured at n = 2^22, theta 0.75 (55 a
        # level of log2 n), growing as theta^-3 in the usual way; 66
        # operations with the quadrupole, 22 without
        per = 55.0 * math.log2(n) * (0.75 / case["theta"]) ** 3
        return dict(bytes=(16 + 4 + 12) * n + 80 * 4.0 * n / case["n_crit"],
                    flops=min(per, n) * n * (60.0 if case["quad"] else 22.0))
    if kind == "reorder":
        return dict(bytes=(4 * 4 + 2 * (12 + 12 + 4 + 8)) * n, flops=0)
    return dict(bytes=(12 + 12) * n, flops=30.0 * n)


def tolerance(case):
    kind = case["kind"]
    if kind in ("reorder", "noalloc"):
        return "exact"
    if kind == "walk":
        # FP32 sums of about a thousand terms of both signs, and a cell here
        # and there whose opening test is a tie to rounding
        return {"rel": 1e-5, "max": 1e-3}
    # integers equal; the second moments are up to 2.8e-6 off their 64-bit
    # values (the norm is that of the largest cells, which sum over all
    # levels), masses and centres 2e-7
    return {"rel": 1e-5, "max": 1e-4}


# ------------------------------------------------------------------ exact

def _keys(pos, lo, side, hilbert):
    """The 63 key bits below the leading 1, int64."""
    q = ((pos - lo) * (2097152.0 / side)[:, None] if side.dim() else (pos - lo) * (2097152.0 / side))
    q = q.floor_().clamp_(0.0, 2097151.0).to(torch.int64)
    x, y, z = q[:, 0].clone(), q[:, 1].clone(), q[:, 2].clone()
    del q
    if hilbert:
        # Skilling's transform (AIP Conf. Proc. 707, 381, 2004)
        ax = [x, y, z]
        for lev in range(20, 0, -1):
            p = (1 << lev) - 1
            for i in range(3):
                on = (ax[i] >> lev) & 1 == 1
                t = torch.where(on, 0, (ax[0] ^ ax[i]) & p)
                ax[0] ^= torch.where(on, p, t)
                if i:
                    ax[i] ^= t
        ax[1] ^= ax[0]
        ax[2] ^= ax[1]
        t = torch.zeros_like(x)
        for lev in range(20, 0, -1):
            t ^= torch.where((ax[2] >> lev) & 1 == 1, (1 << lev) - 1, 0)
        x, y, z = ax[0] ^ t, ax[1] ^ t, ax[2] ^ t
    key = torch.zeros_like(x)
    for b in range(20, -1, -1):
        key = (key << 3) | (((x >> b) & 1) << 2) | (((y >> b) & 1) << 1) | ((z >> b) & 1)
    return key


def _exact_trees(pos, mass, off, n_crit, hilbert, pow2):
    """Trees of the sets off[s] .. off[s+1] in 64 bits: arrays of the cells
    (set by set, level by level, in key order) and of the particles."""
    n, sets = pos.shape[0], off.numel() - 1
    which = torch.repeat_interleave(torch.arange(sets, device=DEV), torch.diff(off), output_size=n)
    if sets > 1:
        idx = which[:, None].expand(n, 3)
        lo = torch.full((sets, 3), math.inf, device=DEV, dtype=F64).scatter_reduce_(0, idx, pos, "amin")
        hi = torch.full((sets, 3), -math.inf, device=DEV, dtype=F64).scatter_reduce_(0, idx, pos, "amax")
    else:
        lo, hi = pos.amin(0, keepdim=True), pos.amax(0, keepdim=True)
    side = (hi - lo).amax(1)
    side = torch.where(side > 0, side, 1.0)
    if pow2:
        m, e = torch.frexp(side)
        side = torch.where(m == 0.5, side, torch.ldexp(torch.ones_like(side), e))
    root = torch.cat([lo, side[:, None]], dim=1)
    if sets > 1:
        key = _keys(pos, lo[which], side[which], hilbert)
    else:
        key = _keys(pos, lo[0], side[0], hilbert)
    key, perm = torch.sort(key, stable=True)
    if sets > 1:
        w, order = torch.sort(which[perm], stable=True)
        key, perm = key[order], perm[order]
    del which
    pos, mass = pos[perm], mass[perm]
    # cells, level by level: segments of equal key prefixes inside split cells
    pf, pe = off[:-1], off[1:]
    keep = pe > pf
    pf, pe, cset = pf[keep], pe[keep], torch.arange(sets, device=DEV)[keep]
    levels = [dict(pf=pf, pe=pe, set=cset, par=torch.full_like(pf, -1))]
    starts = torch.zeros(n, dtype=torch.bool, device=DEV)
    starts[pf] = True
    for d in range(1, 22):
        up = levels[-1]
        if not bool((up["pe"] - up["pf"] > n_crit).any()):
            break
        pre = key >> (63 - 3 * d)
        starts[1:] |= pre[1:] != pre[:-1]
        del pre
        pf = starts.nonzero().squeeze(1)
        pe = torch.cat([pf[1:], pf.new_tensor([n])])
        par = torch.searchsorted(up["pf"], pf, right=True) - 1
        ok = par >= 0
        par.clamp_(min=0)
        ok &= (pf < up["pe"][par]) & (up["pe"][par] - up["pf"][par] > n_crit)
        pf, pe, par = pf[ok], pe[ok], par[ok]
        levels.append(dict(pf=pf, pe=pe, set=up["set"][par], par=par))
    # moments: leaves from their members, other cells from their children
    below = None
    for d in range(len(levels) - 1, -1, -1):
        c = levels[d]
        k = c["pf"].numel()
        M = torch.zeros(k, device=DEV, dtype=F64)
        S = torch.zeros(k, 3, device=DEV, dtype=F64)
        Q = torch.zeros(k, 6, device=DEV, dtype=F64)
        b = torch.full((k, 6), math.inf, device=DEV, dtype=F64)
        b[:, 3:] = -math.inf
        cnt = c["pe"] - c["pf"]
        leaf = (cnt <= n_crit) if d < 21 else torch.ones_like(cnt, dtype=torch.bool)
        ref = pos[c["pf"]]

        def add(i, m, x, q, box):
            r = x - ref[i]
            M.index_add_(0, i, m)
            S.index_add_(0, i, m[:, None] * r)
            w = torch.stack([r[:, a] * r[:, e] for a in range(3) for e in range(a, 3)], dim=1).mul_(m[:, None])
            Q.index_add_(0, i, w if q is None else w.add_(q))
            j = i[:, None].expand(-1, 3)
            b[:, :3] = b[:, :3].scatter_reduce(0, j, box[:, :3], "amin")
            b[:, 3:] = b[:, 3:].scatter_reduce(0, j, box[:, -3:], "amax")

        li = leaf.nonzero().squeeze(1)
        if li.numel():
            lc = cnt[li]
            tot = int(lc.sum())
            i = torch.repeat_interleave(li, lc, output_size=tot)
            first = torch.cumsum(lc, 0) - lc
            p = torch.arange(tot, device=DEV) - torch.repeat_interleave(first - c["pf"][li], lc, output_size=tot)
            add(i, mass[p], pos[p], None, pos[p])
            del i, p
        if below is not None:
            add(below["par"], below["M"], below["com"], below["Q"], below["box"])
        r = torch.where(M[:, None] != 0, S / M[:, None], 0.0)
        w = torch.stack([r[:, a] * r[:, e] for a in range(3) for e in range(a, 3)], dim=1)
        c.update(M=M, com=ref + r, Q=Q - M[:, None] * w, box=b)
        below = c
    cat = {k: torch.cat([c[k] for c in levels]) for k in ("M", "com", "Q", "box", "set")}
    order = torch.sort(cat["set"], stable=True)[1] if sets > 1 else slice(None)
    cells = dict(mass=cat["M"][order], com=cat["com"][order], quad=cat["Q"][order], aabb=cat["box"][order])
    return cells, torch.cat([pos, mass[:, None]], dim=1), root


def exact(case, seed):
    kind = case["kind"]
    if kind in ("reorder", "noalloc"):
        return None
    pos, mass, off = _inputs(case, seed)
    if kind == "walk":
        if case["n"] > 20000:
            return None   # the direct sum in 64 bits takes too long
        # the sum the walk approximates, softened as it is
        x = pos.to(F64)
        eps2 = (1e-3 * float((x.amax(0) - x.amin(0)).amax())) ** 2
        m = mass.to(F64)
        acc = torch.empty_like(x)
        for a in range(0, x.shape[0], 512):
            r = x[None, :, :] - x[a:a + 512, None, :]
            w = m * (r.square().sum(2) + eps2) ** -1.5
            acc[a:a + 512] = (w[:, :, None] * r).sum(1)
        return acc
    n = pos.shape[0]
    if mass is None:
        mass = torch.full((n,), 1.0 / n, device=DEV, dtype=torch.float32)
    single = off is None
    if single:
        off = torch.tensor([0, n], device=DEV)
    cells, srt, root = _exact_trees(pos.to(F64), mass.to(F64), off, case["n_crit"],
                                    case.get("key") == "hilbert",
                                    bool(case.get("pow2")))
    if case.get("pair"):
        cells["centre"] = cells["com"]
    if case.get("mode") == "fp64":
        cells.update(mass64=cells["mass"], com64=cells["com"], quad64=cells["quad"])
    # the arrays' whole lengths, clear past the last cell
    more = _capacity(case, n) - cells["mass"].shape[0]
    out = {k: torch.cat([v, v.new_zeros(more, *v.shape[1:])]) for k, v in cells.items()}
    for k in ("pkey", "perm", "ckey", "level", "parent", "child_first", "child_end", "pfirst",
              "pend", "leaf_cell"):
        out[k] = None
    if not single:
        out.update(set_cell_offset=None, set_root=root)
    if case.get("sorted_pos"):
        out["pos_sorted"] = srt
    return out
