"""Performance cases of the CompaSO hot path, as a program calls it.

A case names a seeded particle set, the context's options and the entry point
that takes it: ``cso_find_groups`` on device or host buffers, the three steps
one at a time, the served queue, and the slab stream.  Particle sets follow
the recipes of ``paper_2110_11408_gb300/synth.py`` (uniform background plus
truncated NFW haloes with power-law sizes, or pre-formed isolated groups),
drawn on the GPU here so that the big ones are made quickly.

Every output is a whole number, or a catalogue row handed over as its bytes:
kernel sums, labels and rows are decided in exact integers, so nothing here
has a rounding error to measure.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2110_11408_gb300 import cso

BOX = 1 << 21
FOUR_PI_3 = 4.0 * math.pi / 3.0


def listed():
    return [
        # the smallest request a program sends (the smoke run's patch across the
        # periodic corner): launches and host round trips are most of the time
        dict(name="patch", kind="box", u=32768, ext=16.0, recipe="small", flags="plain", z=-1.0),
        # one whole box of side 64 on default flags: a coarse box of 262,144 particles
        dict(name="tiny", kind="box", u=32768, ext=0.0, recipe="small", flags="plain", z=-1.0),
        # the same size as a script calls it: numpy buffers in and out, radial statistics asked for
        dict(name="tiny-host", kind="host", u=32768, ext=0.0, recipe="small", flags="batched", z=-1.0),
        # a box of side 128 on the batched schedule: the size of one served request
        dict(name="box128", kind="box", u=16384, ext=0.0, recipe="medium", flags="batched", z=-1.0),
        # the same with radial statistics and shrinking-sphere centres, thresholds at z = 0.5
        dict(name="box128-radial", kind="radial", u=16384, ext=0.0, recipe="medium", flags="batched", z=0.5),
        # the headline box: side 256, 16.8M particles, batched
        dict(name="medium", kind="box", u=8192, ext=0.0, recipe="medium", flags="batched", z=-1.0),
        # a large fine box, a side that is no power of two: 64M particles, 10^9 cells
        dict(name="large", kind="box", u=5243, ext=0.0, recipe="medium", flags="batched", z=-1.0),
        # pre-formed groups of uneven size, one of 2 million particles among thousands of small ones
        dict(name="uneven-groups", kind="groups", u=8192, n=4_000_000, giant=2_000_000, nmin=35, nmax=2_000_000,
             subs=5, flags="batched"),
        # very many small groups of nearly one size
        dict(name="many-groups", kind="groups", u=8192, n=4_000_000, giant=0, nmin=35, nmax=45, subs=0,
             flags="batched"),
        # a rank of a distributed run: density, FoF and levels as three calls on device buffers
        dict(name="steps", kind="steps", u=16384, ext=0.0, recipe="medium", flags="batched", z=-1.0),
        # a box delivered as x-slabs, ghosts and open groups kept between them
        dict(name="slab-stream", kind="stream", u=16384, ext=0.0, recipe="medium", flags="batched", z=-1.0, parts=8),
        # independent boxes in the served queue, four at a time
        dict(name="served-boxes", kind="served", u=32768, ext=0.0, recipe="small", flags="batched", z=-1.0, parts=8),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "radial", "host", "steps", "stream", "served", "groups"])
    if kind == "groups":
        n = int(_log_uniform(rng, 3e4, 4e6))
        few = rng.random() < 0.3
        return dict(kind=kind, u=rng.randrange(8192, 12000), n=n,
                    giant=0 if few else int(n * rng.uniform(0.05, 0.5)), nmin=rng.randrange(20, 50),
                    nmax=rng.randrange(60, 400) if few else max(1000, n // 4), subs=0 if few else rng.randrange(6),
                    flags="plain" if n < 200_000 and rng.random() < 0.3 else "batched")
    # grid units per mean spacing: boxes from the coarsest that bins to side 256, odd sides included
    top = 1 << 23 if kind == "box" else 1 << 21
    u = int(_log_uniform(rng, max(8192, 1.01 * BOX / top ** (1 / 3)), 40000))
    side = BOX / u
    ext = 0.0 if rng.random() < 0.6 else round(_log_uniform(rng, 10.0, 0.9 * side), 3)
    case = dict(kind=kind, u=u, ext=ext, recipe=rng.choice(["small", "medium"]),
                flags="plain" if rng.random() < 0.25 else "batched",
                z=-1.0 if rng.random() < 0.7 else round(rng.uniform(0.0, 3.0), 3))
    if kind in ("stream", "served"):
        case["parts"] = rng.randrange(3, 9)
    return case


# --------------------------------------------------------------------------
# particle sets
# --------------------------------------------------------------------------
RECIPES = {  # background share, halo sizes, share of hosts with a satellite
    "small": (0.5, 20, 20_000, 0.0),
    "medium": (0.4, 20, 200_000, 0.1),
}


def _r200(n):
    return (np.asarray(n, np.float64) / (200.0 * FOUR_PI_3)) ** (1.0 / 3.0)


def _isotropic(gen, n):
    z = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * 2.0 - 1.0
    phi = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    s = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], dim=1)


def _nfw_points(gen, centres, sizes, conc, u):
    """Particles of NFW haloes truncated at R_200, grid units (not wrapped)."""
    sizes = torch.as_tensor(sizes, device="cuda")
    k = torch.repeat_interleave(torch.arange(sizes.numel(), device="cuda"), sizes)
    c = torch.as_tensor(conc, device="cuda")[k]
    mu = lambda y: torch.log1p(y) - y / (1.0 + y)  # noqa: E731
    q = torch.rand(k.numel(), generator=gen, device="cuda", dtype=torch.float64) * mu(c)
    lo, hi = torch.zeros_like(q), torch.ones_like(q)
    for _ in range(36):
        mid = 0.5 * (lo + hi)
        below = mu(c * mid) < q
        lo = torch.where(below, mid, lo)
        hi = torch.where(below, hi, mid)
    rad = 0.5 * (lo + hi) * torch.as_tensor(_r200(sizes.cpu().numpy()), device="cuda")[k] * u
    return torch.as_tensor(centres, device="cuda")[k] + rad[:, None] * _isotropic(gen, k.numel())


def _finish(gen, parts):
    """Grid positions int32 [n, 3] and ids int64 [n], in a seeded shuffled order."""
    p = torch.cat(parts)
    pos = torch.remainder(torch.round(p).to(torch.int64), BOX).to(torch.int32)
    perm = torch.randperm(p.shape[0], generator=gen, device="cuda")
    return pos[perm].contiguous(), perm.contiguous()


def _box_particles(case, seed):
    """A whole box at the mean density (ext = 0), or a cube of `ext` mean
    spacings of one, straddling the periodic corner."""
    frac_bg, nmin, nmax, sat = RECIPES[case["recipe"]]
    u, rng = case["u"], np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ext = case["ext"] or BOX / u
    lo = -0.5 * case["ext"]
    n = int(round(ext ** 3))
    budget = n - int(round(frac_bg * n))
    a = -0.9  # dN/dN ~ N^-1.9
    sizes, ratio, used = [], [], 0
    while used < budget:
        s = np.floor((nmin ** a + rng.random(4096) * (float(nmax) ** a - nmin ** a)) ** (1.0 / a)).astype(np.int64)
        r = np.where(rng.random(4096) < sat, rng.uniform(0.05, 0.3, 4096), 0.0)
        sizes.append(s)
        ratio.append(r)
        used += int(s.sum() + np.rint(s * r).sum())
    sizes, ratio = np.concatenate(sizes), np.concatenate(ratio)
    small = np.rint(sizes * ratio).astype(np.int64)
    small[small < nmin] = 0
    keep = np.cumsum(sizes + small) <= budget
    sizes, small = sizes[keep], small[keep]
    centres = (lo + rng.random((sizes.size, 3)) * ext) * u
    w = small > 0
    v = rng.normal(size=(int(w.sum()), 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    sub = centres[w] + (rng.uniform(0.3, 1.5, len(v)) * _r200(sizes[w]) * u)[:, None] * v
    centres, all_sizes = np.concatenate([centres, sub]), np.concatenate([sizes, small[w]])
    parts = []
    if all_sizes.size:
        parts.append(_nfw_points(gen, centres, all_sizes, rng.uniform(4.0, 12.0, all_sizes.size), u))
    n_bg = n - int(all_sizes.sum())
    parts.append((torch.rand(n_bg, 3, generator=gen, device="cuda", dtype=torch.float64) * ext + lo) * u)
    return _finish(gen, parts)


def _group_particles(case, seed):
    """Isolated pre-formed groups without background: sizes with equal
    particles per logarithmic interval (and one giant), each a host with up to
    `subs` subhaloes.  Groups wider than 4 mean spacings are shelved side by
    side from z = 0 up, the others take random sites of a lattice above them."""
    u, rng = case["u"], np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nmin, nmax, side = case["nmin"], case["nmax"], BOX / case["u"]
    sizes = [np.array([case["giant"]] if case["giant"] else [], np.int64)]
    used = case["giant"]
    while used < case["n"]:
        s = np.floor(1.0 / (1.0 / nmin - rng.random(4096) * (1.0 / nmin - 1.0 / nmax))).astype(np.int64)
        sizes.append(s)
        used += int(s.sum())
    sizes = np.concatenate(sizes)
    sizes = np.sort(sizes[np.cumsum(sizes) <= case["n"]])[::-1].copy()
    sizes[: case["n"] - int(sizes.sum())] += 1
    sizes[0] += case["n"] - int(sizes.sum())  # n particles for every seed
    G = sizes.size
    nsub = rng.integers(0, case["subs"] + 1, G) if case["subs"] else np.zeros(G, np.int64)
    owner = np.repeat(np.arange(G), nsub)
    ratio = rng.uniform(0.01, 0.3, owner.size)
    host = sizes / (1.0 + np.bincount(owner, ratio, minlength=G))
    sub = np.rint(ratio * host[owner]).astype(np.int64)
    ok = sub >= 20
    owner, sub = owner[ok], sub[ok]
    hosts = sizes - np.bincount(owner, sub, minlength=G).astype(np.int64)
    dist = rng.uniform(0.2, 0.9, owner.size) * _r200(hosts[owner])
    reach = _r200(hosts)
    np.maximum.at(reach, owner, dist + _r200(sub))
    reach += 0.3  # half the gap between two groups' spheres: wider than b and l_FoF
    centres = np.zeros((G, 3))
    x = y = z = row = layer = 0.0
    wide = int(np.searchsorted(-sizes, -int(200 * FOUR_PI_3 * 1.2 ** 3)))
    while wide < G and reach[wide:].max() > 2.0:
        wide += 1
    for g in range(wide):
        d = 2.0 * reach[g]
        if x + d > side:
            x, y, row = 0.0, y + row, 0.0
        if y + d > side:
            x, y, z, row, layer = 0.0, 0.0, z + layer, 0.0, 0.0
        centres[g] = (x + reach[g], y + reach[g], z + reach[g])
        x, row, layer = x + d, max(row, d), max(layer, d)
    z += layer
    if wide < G:
        pitch = 2.0 * reach[wide:].max()
        m, mz = int(side // pitch), int((side - z) // pitch)
        site = rng.choice(m * m * mz, G - wide, replace=False)
        centres[wide:] = np.stack([site % m, site // m % m, site // (m * m)], axis=1) * pitch + 0.5 * pitch
        centres[wide:, 2] += z
    v = rng.normal(size=(owner.size, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    all_c = np.concatenate([centres, centres[owner] + dist[:, None] * v]) * u
    all_n = np.concatenate([hosts, sub])
    return _finish(gen, [_nfw_points(gen, all_c, all_n, rng.uniform(4.0, 12.0, all_n.size), u)])


# --------------------------------------------------------------------------
# states: one context per set of options lives as long as the process, as a
# program that handles box after box keeps it
# --------------------------------------------------------------------------
_contexts = {}


def _context(case):
    flags = 0 if case["flags"] == "plain" else cso.FLAG_BATCHED
    if case["kind"] == "served":
        flags |= cso.FLAG_SLOTS(4)
    if case["kind"] == "stream":
        flags |= cso.FLAG_SLOTS(2)
    if flags not in _contexts:
        _contexts[flags] = cso.Context(0, flags=flags)
    return _contexts[flags]


_stream_ids = [0]


def prepare(case, seed):
    s = _state(case, seed)
    torch.cuda.synchronize()  # the library's streams do not wait for torch's
    return s


def _state(case, seed):
    kind = case["kind"]
    p = cso.cso_params_default(case["u"])
    if case.get("z", -1.0) >= 0.0:
        cso.cso_params_cosmology(p, 0.315, case["z"])
    s = dict(kind=kind, ctx=_context(case), params=p)
    if kind == "groups":
        s["buffers"] = _buffers(*_group_particles(case, seed))
        return s
    if kind == "served":
        s["buffers"] = [_buffers(*_box_particles(case, seed * 16 + k)) for k in range(case["parts"])]
        return s
    pos, ids = _box_particles(case, seed)
    n = pos.shape[0]
    if kind == "host":
        s["buffers"] = _buffers(pos.cpu().numpy(), ids.cpu().numpy().view(np.uint64),
                                want=("l0", "l1", "l2", "sigma", "radial"))
    elif kind == "steps":
        s["pos"], s["ids"], s["n"] = pos, ids, n
        s["sigma"], s["l0"], s["l1"], s["l2"] = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(4))
        s["cap"] = max(16, n // 35 + 1)
        s["halos"] = torch.zeros(s["cap"] * cso.HALO_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    elif kind == "stream":
        edges = [BOX * k // case["parts"] for k in range(case["parts"] + 1)]
        slab = torch.bucketize(pos[:, 0].contiguous(), torch.tensor(edges[1:-1], device="cuda", dtype=torch.int32),
                               right=True)
        # the slabs' labels and sums are slices of the whole box's
        s["out"] = {name: torch.empty(n, dtype=torch.int64, device="cuda") for name in ("l0", "l1", "l2", "sigma")}
        s["halos"] = torch.zeros(n // 20 + 64, cso.HALO_DTYPE.itemsize // 8, dtype=torch.int64, device="cuda")
        s["buffers"], at = [], 0
        for k in range(case["parts"]):
            m = slab == k
            b = cso.Buffers(pos[m].contiguous(), ids[m].contiguous(), True, halo_cap=n // 20 + 64, want=(),
                            x_lo=edges[k], x_hi=edges[k + 1])
            for name, whole in s["out"].items():
                b.out[name] = whole[at:at + b.n]
                setattr(b.cout, name, b.out[name].data_ptr())
            at += b.n
            s["buffers"].append(b)
    else:
        s["buffers"] = _buffers(pos, ids, want=("l0", "l1", "l2", "sigma") + (("radial",) if kind == "radial" else ()))
    return s


def _buffers(pos, ids, want=("l0", "l1", "l2", "sigma")):
    """A request's buffers; catalogue rows past the last one found stay zero."""
    b = cso.Buffers(pos, ids, not isinstance(pos, np.ndarray), want=want)
    for rows in (b.halos, b.radial):
        if isinstance(rows, np.ndarray):
            rows.view(np.uint8)[:] = 0
        elif rows is not None:
            rows.zero_()
    return b


def _outputs(b):
    """The result as it lies in the request's own buffers."""
    r = dict(b.out, halos=b.halos, n_halos=int(b.cout.n_halos))
    if b.radial is not None:
        r["radial"] = b.radial
    if not b.out_device:
        r = {k: v.view(np.uint8 if k in ("halos", "radial") else np.int64) if k != "n_halos" else v
             for k, v in r.items()}
    return r


def _queue(ctx, buffers, params):
    tickets = [ctx.submit(b, params) for b in buffers]
    for t in tickets:
        done, rc = ctx.wait(t)
        if not done or rc != cso.CSO_OK:
            raise cso.CsoError(rc, "served request")


def run(state):
    kind, ctx, p = state["kind"], state["ctx"], state["params"]
    if kind == "served":
        _queue(ctx, state["buffers"], p)
        return [_outputs(b) for b in state["buffers"]]
    if kind == "stream":
        _stream_ids[0] += 1
        for b in state["buffers"]:
            b.cin.request_id = _stream_ids[0]
        _queue(ctx, state["buffers"], p)
        # the box's catalogue: every slab's rows (unordered) by nucleus id
        size = cso.HALO_DTYPE.itemsize
        rows = torch.cat([b.halos[: int(b.cout.n_halos) * size] for b in state["buffers"]])
        rows = rows.view(torch.int64).view(-1, size // 8)
        torch.index_select(rows, 0, torch.argsort(rows[:, 0]), out=state["halos"][: rows.shape[0]])
        return dict(state["out"], halos=state["halos"], n_halos=rows.shape[0])
    if kind == "steps":
        lib, n, ref = cso.lib(), state["n"], ctypes.byref(p)
        ptr = {k: state[k].data_ptr() for k in ("pos", "ids", "sigma", "l0", "l1", "l2", "halos")}
        out = cso.CsoOutput(l1=ptr["l1"], l2=ptr["l2"], halos=ptr["halos"], halo_cap=state["cap"], on_device=1)
        for name, rc in (
                ("cso_density", lib.cso_density(ctx.h, ptr["pos"], n, n, ref, ptr["sigma"], 1)),
                ("cso_fof", lib.cso_fof(ctx.h, ptr["pos"], ptr["ids"], ptr["sigma"], n, ref, ptr["l0"], 1)),
                ("cso_levels", lib.cso_levels(ctx.h, ptr["pos"], ptr["ids"], ptr["sigma"], ptr["l0"], n, ref,
                                              ctypes.byref(out)))):
            if rc != cso.CSO_OK:
                raise cso.CsoError(rc, name)
        r = {k: state[k] for k in ("sigma", "l0", "l1", "l2")}
        return dict(r, halos=state["halos"], n_halos=out.n_halos)
    cso.cso_find_groups(ctx.h, state["buffers"], p)
    return _outputs(state["buffers"])


def work(case):
    """Bytes: positions and ids once in, the four per-particle outputs once
    out.  Operations: 11 integer ones per pair of particles within b, about
    290 such pairs per particle in these recipes (counted on the side-256
    box)."""
    if case["kind"] == "groups":
        n = case["n"]
    else:
        n = int(round((case["ext"] or BOX / case["u"]) ** 3)) * (case["parts"] if case["kind"] == "served" else 1)
    return {"bytes": n * (12 + 8 + 32), "flops": n * 290 * 11}
