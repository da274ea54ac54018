"""The workloads this library's speed is judged on.

Each case is one call (or one short sequence of calls) a program makes of the
public Python binding, `paper_0904_3662_gb300.ahf`, on synthetic haloes of the
laws `synth` documents, drawn on the GPU from a seed.  A case is a dict of
plain values:

  kind      which entry points a pass calls (see `run`)
  haloes    number of haloes (hosts for the kinds of large hosts)
  lo, hi    range of the particle counts, N_p ~ N_p^-1.9 on [lo, hi]
  cont      background particles per halo particle
  coord     "f32" relative to the centre, "f64" absolute, "box" float32 in a
            periodic box
  fp64      the all-FP64 mode (else mixed precision)
  masses    per-particle masses (else one mass for all)
  gas       a thermal energy per particle
  bins      profile bins (0: no profile)
  variant   ahf_params.variant bits

`exact` is a plain torch FP64 evaluation of the method, vectorised over the
haloes of a case.
"""
import math

import numpy as np
import torch

from paper_0904_3662_gb300 import ahf, synth

N_SUB = 20                # subhaloes of a large host
SUB_FRAC = 0.005          # particles of each, as a fraction of the host's
BOX = 5e5
R_MIN_FRAC = 0.01
EXACT_MAX = 30_000_000    # candidates above which `exact` would take too long


def _case(name, kind, haloes, lo, hi, cont=0.15, coord="f32", fp64=False, masses=False, gas=False, bins=0, variant=0):
    return {"name": name, "kind": kind, "haloes": haloes, "lo": lo, "hi": hi, "cont": cont, "coord": coord,
            "fp64": fp64, "masses": masses, "gas": gas, "bins": bins, "variant": variant}


def listed():
    return [
        # one small halo as it arrives, alone: launches and latency
        _case("request_317", "unbind", 1, 276, 276),
        # the 10,000-particle halo with 1,000 background particles, float64
        # positions, mixed precision, with its profile
        _case("halo_11k", "unbind_profile", 1, 10_000, 10_000, cont=0.1, coord="f64", bins=32),
        # the same halo in the all-FP64 mode
        _case("halo_11k_fp64", "unbind_profile", 1, 10_000, 10_000, cont=0.1, coord="f64", fp64=True, bins=32),
        # the benchmark's batch of 2,000 haloes of 1e2 to 1e5 particles
        _case("batch_2000", "unbind_profile", 2000, 100, 100_000, bins=32),
        # the same batch from and to page-locked host memory (a catalogue
        # code whose particles live on the host)
        _case("host_2000", "host", 2000, 100, 100_000, bins=32),
        # a whole snapshot's haloes, float64 positions (a fifth of the
        # precision sweep's 100,000)
        _case("sweep_20000", "unbind", 20_000, 100, 100_000, cont=0.1, coord="f64"),
        # part of the same population in the all-FP64 mode
        _case("sweep_3000_fp64", "unbind", 3000, 100, 100_000, cont=0.1, coord="f64", fp64=True),
        # the large-halo tail: 64 hosts of 1e6 to 1e7 particles with 20
        # subhaloes each, float32 coordinates in a periodic box, with profiles
        _case("tail_64", "unbind_profile", 64, 1_000_000, 10_000_000, cont=0.0, coord="box", bins=32),
        # a few hosts of a zoom simulation with gas: a mass and a thermal
        # energy per particle
        _case("gas_3", "unbind", 3, 1_000_000, 3_000_000, cont=0.0, coord="box", masses=True, gas=True),
        # a finished catalogue's post-processing: profiles of 64 bins,
        # spins and energies, and the cross-match against a second catalogue
        _case("catalogue_1500", "catalogue", 1500, 100, 100_000, bins=64),
        # hosts of a multi-mass zoom with 20 subhaloes each, subhaloes
        # unbound first, shared particles through member lists
        _case("hierarchy_9", "hierarchy", 9, 20_000, 200_000, cont=0.0, coord="box", masses=True),
        # a burst of requests to the serving layer, submitted one by one
        # from host memory and polled until each is done
        _case("serve_200", "serve", 200, 100, 100_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["request", "halo", "halo", "batch", "batch", "host", "sweep", "sweep", "tail", "gas",
                       "catalogue", "hierarchy", "serve"])
    if kind == "request":
        n = _log_int(rng, 100, 100_000)
        return _drop(_case("", "unbind", 1, n, n, cont=round(rng.uniform(0.0, 0.3), 3)))
    if kind == "halo":
        n = _log_int(rng, 500, 200_000)
        return _drop(_case("", "unbind_profile", 1, n, n, cont=0.1, coord=rng.choice(["f64", "f32"]),
                           fp64=rng.random() < 0.5, bins=rng.choice([16, 32, 50])))
    if kind == "batch":
        return _drop(_case("", rng.choice(["unbind", "unbind_profile"]), _log_int(rng, 8, 4000), 100,
                           _log_int(rng, 1000, 100_000), coord=rng.choice(["f32", "f64"]),
                           masses=rng.random() < 0.3, bins=rng.choice([20, 32, 64]),
                           variant=rng.choice([0, 0, ahf.VAR_VBULK_INITIAL])))
    if kind == "host":
        return _drop(_case("", "host", _log_int(rng, 50, 4000), 100, 100_000, bins=32,
                           coord=rng.choice(["f32", "f64"])))
    if kind == "sweep":
        fp64 = rng.random() < 0.5
        return _drop(_case("", "unbind", _log_int(rng, 200, 3000) if fp64 else _log_int(rng, 2000, 20_000), 100,
                           100_000, cont=0.1, coord="f64", fp64=fp64))
    if kind == "tail":
        hi = _log_int(rng, 500_000, 10_000_000)
        return _drop(_case("", "unbind_profile", _log_int(rng, 1, 32), hi // 4, hi, cont=0.0, coord="box", bins=32,
                           masses=rng.random() < 0.25))
    if kind == "gas":
        hi = _log_int(rng, 20_000, 3_000_000)
        return _drop(_case("", "unbind", rng.randint(1, 4), hi // 3, hi, cont=0.0, coord="box",
                           masses=rng.random() < 0.7, gas=True))
    if kind == "catalogue":
        return _drop(_case("", "catalogue", _log_int(rng, 20, 2000), 100, 100_000, bins=rng.choice([32, 64, 200])))
    if kind == "hierarchy":
        return _drop(_case("", "hierarchy", _log_int(rng, 1, 12), 20_000, _log_int(rng, 50_000, 200_000), cont=0.0,
                           coord="box", masses=rng.random() < 0.5))
    return _drop(_case("", "serve", _log_int(rng, 20, 300), 100, _log_int(rng, 1000, 100_000)))


def _drop(c):
    del c["name"]
    return c


# ---- inputs ----------------------------------------------------------------------

_TABLES = {}


def _tables():
    """Inverse mass function x(u)/x_t and velocity dispersion (in sqrt(G M_s / r_s))
    of truncated NFW spheres, over a grid of ln c: x_t = 2c, and x_t = c for
    subhaloes."""
    if not _TABLES:
        lnc = np.linspace(math.log(3.0), math.log(45.0), 40)
        for trunc in (1.0, 2.0):
            inv, sig = [], []
            for c in np.exp(lnc):
                x_t = trunc * c
                x = np.geomspace(1e-7 * x_t, x_t, 2048)
                m = synth.m_nfw(x)
                inv.append(np.interp(np.linspace(0.0, 1.0, 4097), m / m[-1], x) / x_t)
                f = m / (x ** 2 * (1.0 + x) ** 2)
                seg = 0.5 * (f[1:] + f[:-1]) * np.diff(np.log(x))
                tail = np.concatenate([np.cumsum(seg[::-1])[::-1], [0.0]])
                s2 = x * (1.0 + x) ** 2 * tail
                # on a grid of ln(x / x_t), -16 to 0
                sig.append(np.sqrt(np.interp(np.linspace(-16.0, 0.0, 1025), np.log(x / x_t), s2)))
            _TABLES[trunc] = (torch.from_numpy(np.stack(inv)).cuda(), torch.from_numpy(np.stack(sig)).cuda())
        _TABLES["lnc"] = (float(lnc[0]), float(lnc[1] - lnc[0]), len(lnc))
    return _TABLES


def _lookup(tab, row, col):
    """Bilinear interpolation of a table at fractional (row, column)."""
    i = row.floor().clamp_(0, tab.shape[0] - 2)
    j = col.floor().clamp_(0, tab.shape[1] - 2)
    a, b = row - i, col - j
    k = i.long() * tab.shape[1] + j.long()
    flat = tab.view(-1)
    top = flat[k] * (1 - b) + flat[k + 1] * b
    bot = flat[k + tab.shape[1]] * (1 - b) + flat[k + tab.shape[1] + 1] * b
    return top * (1 - a) + bot * a


def _nfw(g, c, r200, trunc):
    """Positions and velocities (each a list of 3 tensors) of one particle per
    entry of c, r200 (tensors), drawn from its halo's truncated profile."""
    T = _tables()
    inv, sig = T[trunc]
    l0, dl, nl = T["lnc"]
    n, dev = c.shape[0], c.device
    row = ((c.log() - l0) / dl).clamp_(0, nl - 1)
    f = _lookup(inv, row, torch.rand(n, generator=g, device=dev, dtype=torch.float64) * (inv.shape[1] - 1))
    f.clamp_(min=1e-6)
    rs = r200 / c
    rad = f * trunc * r200
    m200 = (4.0 * math.pi / 3.0 * synth.DELTA_RHO_200C) * r200 ** 3
    ms = m200 / (torch.log1p(c) - c / (1.0 + c))
    s = _lookup(sig, row, (f.log() + 16.0) * ((sig.shape[1] - 1) / 16.0)) * (synth.G_GRAV * ms / rs).sqrt()
    vel = [torch.randn(n, generator=g, device=dev) * s for _ in range(3)]
    return _directions(g, rad), vel


def _directions(g, rad):
    n, dev = rad.shape[0], rad.device
    cth = torch.rand(n, generator=g, device=dev, dtype=torch.float64) * 2 - 1
    ph = torch.rand(n, generator=g, device=dev, dtype=torch.float64) * (2 * math.pi)
    sth = (1 - cth * cth).clamp_(min=0).sqrt()
    return [rad * sth * ph.cos(), rad * sth * ph.sin(), rad * cth]


def _population(case, seed):
    """Particle tensors and host halo arrays of a case.  A case fixes its
    haloes' sizes and concentrations; the seed draws everything else."""
    law = np.random.default_rng(case["haloes"] * 1_000_003 + case["lo"] * 101 + case["hi"])
    rng = np.random.default_rng(seed)
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    nh, coord = case["haloes"], case["coord"]
    counts = synth.powerlaw_counts(law, nh, case["lo"], case["hi"])
    total = counts + np.rint(case["cont"] * counts).astype(np.int64)
    conc = np.exp(np.clip(law.normal(math.log(10.0), 0.25, nh), math.log(4.0), math.log(40.0)))
    offset = np.concatenate([[0], np.cumsum(total)[:-1]]).astype(np.int64)
    hosts = coord == "box"
    own = np.rint(counts * (1.0 - N_SUB * SUB_FRAC)) if hosts else counts
    m200 = own * synth.PARTICLE_MASS * synth.m_nfw(conc) / synth.m_nfw(2.0 * conc)
    r200 = np.array([synth.r200_of_mass(x) for x in m200])
    span = {"f32": 0.0, "f64": 1e5, "box": BOX}[coord]
    centre = rng.uniform(0.0, 1.0, (nh, 3)) * span
    n = int(total.sum())
    dt = torch.float64 if coord == "f64" else torch.float32
    arr = [torch.empty(n, dtype=dt, device=dev) for _ in range(6)]
    mass = torch.empty(n, dtype=dt, device=dev) if case["masses"] else None
    u_th = torch.empty(n, dtype=dt, device=dev) if case["gas"] else None
    subs = []
    # subhaloes: centres drawn from the host's profile inside R_200, bulk
    # velocities N(0, 300 km/s), each truncated at its own R_200
    if hosts:
        n_sub = SUB_FRAC * counts
        sub_r = np.array([synth.r200_of_mass(x * synth.PARTICLE_MASS) for x in n_sub])
        sub_c = np.exp(np.clip(rng.normal(math.log(15.0), 0.25, (nh, N_SUB)), math.log(4.0), math.log(40.0)))
        sub_v = rng.normal(0.0, 300.0, (nh, N_SUB, 3))
        cc = torch.from_numpy(np.repeat(conc, N_SUB)).to(dev)
        rr = torch.from_numpy(np.repeat(r200, N_SUB)).to(dev)
        sub_x = torch.stack(_nfw(g, cc, rr, 1.0)[0], 1).view(nh, N_SUB, 3)
        host_v = rng.normal(0.0, 300.0, (nh, 3))
    # blocks of whole haloes of some 2e7 particles at most (bounded temporaries)
    h0 = 0
    while h0 < nh:
        h1 = h0 + 1
        while h1 < nh and offset[h1] + total[h1] - offset[h0] <= 20_000_000:
            h1 += 1
        lo, hi = int(offset[h0]), int(offset[h1 - 1] + total[h1 - 1])
        hid = torch.repeat_interleave(torch.arange(h0, h1, device=dev), torch.from_numpy(total[h0:h1]).to(dev))
        c = torch.from_numpy(conc).to(dev)[hid]
        r2 = torch.from_numpy(r200).to(dev)[hid]
        pos, vel = _nfw(g, c, r2, 2.0)
        pick = torch.rand(hi - lo, generator=g, device=dev)
        if case["cont"] > 0.0:                      # background particles, mixed among the others
            bg = pick < case["cont"] / (1.0 + case["cont"])
            rad = 2.0 * r2 * torch.rand(hi - lo, generator=g, device=dev, dtype=torch.float64) ** (1.0 / 3.0)
            p2 = _directions(g, rad)
            for a in range(3):
                pos[a] = torch.where(bg, p2[a], pos[a])
                vel[a] = torch.where(bg, torch.randn(hi - lo, generator=g, device=dev).double() * 600.0, vel[a])
        if hosts:                                   # subhalo particles
            at = (pick < N_SUB * SUB_FRAC).nonzero()[:, 0]
            hs = hid[at]
            k = (pick[at] / SUB_FRAC).long().clamp_(max=N_SUB - 1)
            p2, v2 = _nfw(g, torch.from_numpy(sub_c).to(dev)[hs, k], torch.from_numpy(sub_r).to(dev)[hs], 1.0)
            for a in range(3):
                pos[a][at] = p2[a] + sub_x[hs, k, a]
                vel[a][at] = v2[a] + torch.from_numpy(sub_v[:, :, a]).to(dev)[hs, k]
                vel[a] += torch.from_numpy(host_v[:, a].copy()).to(dev)[hid]
        for a in range(3):
            x = pos[a] + torch.from_numpy(centre[:, a].copy()).to(dev)[hid] if span else pos[a]
            if coord == "box":
                x = torch.remainder(x, BOX).to(dt)
                x = torch.where(x >= BOX, torch.zeros_like(x), x)
            arr[a][lo:hi] = x
            arr[3 + a][lo:hi] = vel[a]
        if mass is not None:                        # log-uniform over a decade
            mass[lo:hi] = synth.PARTICLE_MASS * ((torch.rand(hi - lo, generator=g, device=dev) * 2.3 - 1.15).exp())
        if u_th is not None:                        # a third of the particles are gas
            u = torch.rand(hi - lo, generator=g, device=dev)
            u_th[lo:hi] = torch.where(u < 1.0 / 3.0, u * 1.5e5, torch.zeros_like(u))
        del hid, c, r2, pos, vel, pick
        h0 = h1
    parts = ahf.Particles(*arr, mass, synth.PARTICLE_MASS,
                          {"f32": ahf.COORD_F32_REL, "f64": ahf.COORD_F64, "box": ahf.COORD_F32_BOX}[coord], u_th)
    halos = ahf.halo_array(centre, 2.0 * r200, offset, total)
    if hosts:
        subs = [(h, centre[h] + sub_x[h, k].cpu().numpy(), sub_r[h]) for h in range(nh) for k in range(N_SUB)] \
            if case["kind"] == "hierarchy" else []
    return parts, halos, subs


def _params(case):
    return ahf.Params(box=BOX if case["coord"] == "box" else 0.0,
                      precision=ahf.PREC_FP64 if case["fp64"] else ahf.PREC_MIXED, variant=case["variant"])


def _hierarchy(parts, halos, subs):
    """Descriptors, parents and member list of the hosts and their subhaloes: a
    subhalo's candidates are the particles of its host nearest to its centre,
    twice as many as were drawn for it."""
    dev = parts.x.device
    lists, rows, parent = [], [], []
    at = 0
    for h in range(len(halos)):
        n = int(halos["count"][h])
        lists.append(torch.arange(int(halos["offset"][h]), int(halos["offset"][h]) + n, device=dev))
        rows.append((halos["cx"][h], halos["cy"][h], halos["cz"][h], halos["radius"][h], at, n))
        parent.append(-1)
        at += n
    for h, c, r in subs:
        lo = int(halos["offset"][h])
        hi = lo + int(halos["count"][h])
        r2 = 0.0
        for x, cx in zip((parts.x, parts.y, parts.z), c):
            d = x[lo:hi].double() - float(cx)
            d -= BOX * torch.round(d / BOX)
            r2 = r2 + d * d
        n = int(2 * SUB_FRAC * (hi - lo))
        idx = torch.topk(r2, n, largest=False)[1].sort()[0] + lo
        rows.append((c[0], c[1], c[2], r, at, n))
        lists.append(idx)
        parent.append(h)
        at += n
    out = np.zeros(len(rows), dtype=ahf.HALO_DTYPE)
    for k, name in enumerate(("cx", "cy", "cz", "radius", "offset", "count")):
        out[name] = [r[k] for r in rows]
    return out, np.asarray(parent, dtype=np.int64), torch.cat(lists)


_HANDLES = {}


def _context():
    """The program's library handle, kept for its life as a user's program does."""
    if "ctx" not in _HANDLES:
        _HANDLES["ctx"] = ahf.Context(0)
    return _HANDLES["ctx"]


def _server(parts):
    if "serve" not in _HANDLES:
        _HANDLES["serve"] = ahf.Serve(ahf.Params(), device=0, hbm_cap_bytes=2 << 30, coord_type=ahf.COORD_F32_REL,
                                      m0=synth.PARTICLE_MASS)
    return _HANDLES["serve"]


def _records(res):
    """Views of a record buffer: the whole-number fields (n_iter and status
    share one column), M_vir, r_vir and v_bulk."""
    n = res.numel() // ahf.RESULT_DTYPE.itemsize
    f = res.view(torch.float64).view(n, 11)
    return {"ids": res.view(torch.int64).view(n, 11)[:, :6], "m_vir": f[:, 6], "r_vir": f[:, 7], "vbulk": f[:, 8:]}


def _columns(a, n):
    """The columns of a table of different quantities, one view each."""
    return [a[..., k] for k in range(n)]


def _zero_outputs(ctx, n_halos, n_slots, prm):
    out = ctx.alloc_outputs(n_halos, n_slots, precision=prm.precision)
    for t in out.values():
        t.zero_()
    return out


def prepare(case, seed):
    parts, halos, subs = _population(case, seed)
    prm = _params(case)
    kind = case["kind"]
    s = {"kind": kind, "parts": parts, "halos": halos, "prm": prm, "bins": case["bins"], "members": None}
    if kind == "serve":
        s["srv"] = _server(parts)
        host = [t.cpu().numpy() for t in (parts.x, parts.y, parts.z, parts.vx, parts.vy, parts.vz)]
        s["requests"] = []
        for h in halos:
            lo, hi = int(h["offset"]), int(h["offset"] + h["count"])
            one = np.array([h], dtype=ahf.HALO_DTYPE)
            one["offset"] = 0
            p = ahf.Particles(*[np.ascontiguousarray(a[lo:hi]) for a in host], None, synth.PARTICLE_MASS,
                              ahf.COORD_F32_REL)
            s["requests"].append(ahf.Serve.request(p, one))
        s["bound"] = np.zeros(parts.n, dtype=np.int64)
        s["parts"] = None
        return s
    ctx = s["ctx"] = _context()
    if kind == "host":
        keep = []

        def pinned(t):
            t = t.cpu().pin_memory()
            keep.append(t)
            return t.numpy()

        s["keep"] = keep
        s["parts"] = ahf.Particles(*[pinned(t) for t in (parts.x, parts.y, parts.z, parts.vx, parts.vy, parts.vz)],
                                   None, parts.m0, parts.coord_type)
        nh, n = len(halos), parts.n
        res = torch.zeros(nh * ahf.RESULT_DTYPE.itemsize, dtype=torch.uint8)
        s["out"] = {"res": pinned(res), "bound_idx": pinned(torch.zeros(n, dtype=torch.int64)),
                    "phi": pinned(torch.zeros(n)), "removed_iter": pinned(torch.zeros(n, dtype=torch.int32)),
                    "prof": pinned(torch.zeros(nh, case["bins"], 4, dtype=torch.float64))}
        out = s["out"]
        s["result"] = {**_records(torch.from_numpy(out["res"])), "bound": out["bound_idx"], "phi": out["phi"],
                       "removed": out["removed_iter"], "prof": _columns(out["prof"], 4)}
        return s
    if kind == "hierarchy":
        s["halos"], s["parent"], s["members"] = _hierarchy(parts, halos, subs)
    n_slots = ahf.n_slots_of(s["halos"], parts.n, s["members"])
    nh = len(s["halos"])
    out = s["out"] = _zero_outputs(ctx, nh, n_slots, prm)
    rec = _records(out["res"])
    if kind == "catalogue":
        # the catalogue that the pass post-processes, and a second one: the
        # same haloes found again with three in four of their particles
        ctx.unbind_batch(parts, halos, prm, out=out)
        n_b = rec["ids"][:, 0].contiguous()
        off = torch.from_numpy(halos["offset"]).cuda()
        s["match"] = (parts.n, out["bound_idx"], off, n_b, torch.arange(parts.n, device="cuda"),
                      off + torch.from_numpy(halos["count"] // 4).cuda(),
                      torch.from_numpy(halos["count"] - halos["count"] // 4).cuda())
        ctx.sync()
        return s
    s["result"] = {**rec, "bound": out["bound_idx"], "phi": out["phi"], "removed": out["removed_iter"]}
    if kind == "unbind_profile":
        s["prof"] = torch.zeros((nh, case["bins"], 4), dtype=torch.float64, device="cuda")
        s["result"]["prof"] = _columns(s["prof"], 4)
    return s


def run(s):
    kind = s["kind"]
    if kind == "unbind":
        s["ctx"].unbind_batch(s["parts"], s["halos"], s["prm"], out=s["out"])
        return s["result"]
    if kind == "unbind_profile":
        s["ctx"].unbind_profile_batch(s["parts"], s["halos"], s["prm"], n_bins=s["bins"], r_min_frac=R_MIN_FRAC,
                                      out=s["out"], prof=s["prof"])
        return s["result"]
    if kind == "host":
        s["ctx"].unbind_batch_host(s["parts"], s["halos"], s["prm"], out=s["out"], n_bins=s["bins"],
                                   r_min_frac=R_MIN_FRAC)
        return s["result"]
    if kind == "hierarchy":
        s["ctx"].unbind_hierarchy(s["parts"], s["halos"], s["parent"], s["prm"], member_idx=s["members"], out=s["out"])
        return s["result"]
    if kind == "catalogue":
        ctx, out = s["ctx"], s["out"]
        prof = ctx.profile_batch(s["parts"], s["halos"], s["prm"], out["res"], out["bound_idx"], n_bins=s["bins"],
                                 r_min_frac=R_MIN_FRAC)
        props = ctx.halo_properties(s["parts"], s["halos"], s["prm"], out)
        best, shared, xi = ctx.match_catalogs(*s["match"])
        return {"prof": _columns(prof, 4), "props": _columns(props, ahf.PROP_FIELDS), "best": best, "shared": shared,
                "xi": xi}
    srv, done = s["srv"], {}
    ids = []
    for req in s["requests"]:
        rid = srv.submit_prepared(req)
        while rid is None:                          # the ring is full: collect the oldest first
            for i in ids:
                if i not in done:
                    r = srv.poll(i)
                    if r is not None:
                        done[i] = r
                    break
            rid = srv.submit_prepared(req)
        ids.append(rid)
    for i in ids:
        while i not in done:
            r = srv.poll(i)
            if r is not None:
                done[i] = r
    res = np.stack([done[i][0] for i in ids])
    for i, h in zip(ids, s["halos"]):
        b = done[i][1]
        s["bound"][h["offset"]:h["offset"] + len(b)] = b
    return {**_records(torch.from_numpy(res.view(np.uint8))), "bound": s["bound"]}


def work(case):
    """Bytes: the candidates' coordinates and velocities (and masses, thermal
    energies, member lists) once, and per bound particle its index and phi,
    per candidate its removal iteration, per halo its record and rows.  Flops:
    some 25 per particle and iteration (phi, escape test, sums), some 3.5
    iterations."""
    law = np.random.default_rng(case["haloes"] * 1_000_003 + case["lo"] * 101 + case["hi"])
    nh = case["haloes"]
    n = float(synth.powerlaw_counts(law, nh, case["lo"], case["hi"]).sum()) * (1.0 + case["cont"])
    es = 8 if case["coord"] == "f64" else 4
    ps = 8 if case["fp64"] else 4
    per = es * (6 + (1 if case["masses"] else 0) + (1 if case["gas"] else 0))
    if case["kind"] == "catalogue":
        return {"bytes": n * (0.85 * (8 + ps + per) + 16.0) + nh * (88 + 32 * case["bins"] + 96 + 24),
                "flops": 0.85 * n * 60.0}
    if case["kind"] == "hierarchy":
        n *= 1.0 + 2.0 * N_SUB * SUB_FRAC
        per += 8
        nh *= 1 + N_SUB
    bound = 0.85 if case["cont"] > 0 else 0.9
    return {"bytes": n * (per + bound * (8 + ps) + 4) + nh * (88 + 48 + 32 * case["bins"]), "flops": n * 3.5 * 25.0}


# ---- the method in FP64 ----------------------------------------------------------------

def _starts(count):
    return torch.cumsum(count, 0) - count


def _seg_cum(x, start, count):
    """Inclusive prefix sums of x within segments, and the segments' totals."""
    c = torch.cumsum(x, 0)
    base = torch.where(start > 0, c[(start - 1).clamp(min=0)], torch.zeros_like(start, dtype=x.dtype))
    end = torch.where(count > 0, c[(start + count - 1).clamp(min=0)], base)
    return c - torch.repeat_interleave(base, count), end - base


def _unbind(off, vel, m, u_th, hid, nh, radius, prm, keep=None):
    """Candidates off, vel (lists of 3 FP64 tensors), m, u_th in slot order, hid
    their haloes (ascending).  Returns the final sets in (halo, radius) order:
    slots, halo ids, radii, masses, phi, counts, and the sums' v_bulk."""
    dev = hid.device
    r2 = off[0] ** 2 + off[1] ** 2 + off[2] ** 2
    inside = r2 <= (radius * radius)[hid]
    if keep is not None:
        inside &= keep
    slot = inside.nonzero()[:, 0]
    r = r2[slot].sqrt()
    o = torch.sort(r, stable=True)[1]
    o = o[torch.sort(hid[slot][o], stable=True)[1]]
    slot, r = slot[o], r[o]
    h, m = hid[slot], m[slot]
    w = [vel[a][slot] + prm.H * off[a][slot] for a in range(3)]
    v = [vel[a][slot] for a in range(3)]
    u = None if u_th is None else u_th[slot]
    ri = torch.where(r > 0, 1.0 / r, torch.zeros_like(r))
    act = torch.arange(slot.shape[0], device=dev)
    vb = torch.zeros(nh, 3, dtype=torch.float64, device=dev)
    fin, fphi = [], []
    it = 0
    while act.shape[0]:
        it += 1
        ha, ma, ra = h[act], m[act], ri[act]
        cnt = torch.bincount(ha, minlength=nh)
        st = _starts(cnt)
        mi, mt = _seg_cum(ma, st, cnt)
        ti, tt = _seg_cum(ma * ra, st, cnt)
        phi = -prm.G * ((mi - ma) * ra + (tt[ha] - (ti - ma * ra)))
        if it > prm.max_iter:
            fin.append(act)
            fphi.append(phi)
            break
        if it == 1 or not prm.variant & ahf.VAR_VBULK_INITIAL:
            for a in range(3):
                t = _seg_cum(ma * v[a][act], st, cnt)[1] / mt
                vb[:, a] = torch.where(cnt > 0, t, vb[:, a])
        u2 = sum((w[a][act] - vb[ha, a]) ** 2 for a in range(3))
        if u is not None:
            u2 = u2 + 2.0 * u[act]
        gone = u2 > -2.0 * phi
        changed = torch.bincount(ha[gone], minlength=nh) > 0
        done = ~changed[ha]
        fin.append(act[done])
        fphi.append(phi[done])
        act = act[~done & ~gone]
    f = torch.cat(fin)
    phi = torch.cat(fphi)
    f, o = torch.sort(f)
    phi = phi[o]
    cnt = torch.bincount(h[f], minlength=nh)
    st = _starts(cnt)
    mt = _seg_cum(m[f], st, cnt)[1]
    vf = torch.stack([_seg_cum(m[f] * v[a][f], st, cnt)[1] / mt for a in range(3)], 1)
    vf = torch.where((cnt > 0)[:, None], vf, torch.zeros_like(vf))
    return slot[f], h[f], r[f], m[f], phi, cnt, vf


def _virial(h, r, m, cnt, prm):
    """(M_vir, r_vir, k_vir) per halo of sets in (halo, radius) order."""
    st = _starts(cnt)
    nh = cnt.shape[0]
    mi = _seg_cum(m, st, cnt)[0]
    pos = torch.arange(r.shape[0], device=r.device) - st[h]
    rn = torch.cat([r[1:], r.new_full((1,), math.inf)])
    rn = torch.where(pos == cnt[h] - 1, torch.full_like(rn, math.inf), rn)
    crit = prm.delta_rho * 4.0 * math.pi / 3.0
    big = torch.full((nh,), 1 << 60, device=r.device)
    cross = mi < crit * rn ** 3
    k = big.scatter_reduce(0, h[cross], pos[cross], "amin")
    at = (st + torch.where(cnt > 0, k, torch.zeros_like(k))).clamp(max=max(r.shape[0] - 1, 0))
    mv, rk = mi[at], r[at]
    none = (cnt == 0) | (mv < crit * rk ** 3)
    zero = torch.zeros_like(mv)
    return (torch.where(none, zero, mv), torch.where(none, zero, (mv / crit) ** (1.0 / 3.0)),
            torch.where(none, torch.full_like(k, -1), k))


def _rows(h, r, m, cnt, r_vir, n_bins, prm):
    """Profile rows [halo][bin][4]: count, M(<= e), shell density, v_circ."""
    st = _starts(cnt)
    nh = cnt.shape[0]
    mi = torch.cat([r.new_zeros(1), torch.cumsum(m, 0)])
    last = r[(st + cnt - 1).clamp(min=0, max=max(r.shape[0] - 1, 0))]
    r_out = torch.where(r_vir > 0, r_vir, last)
    f = R_MIN_FRAC ** (1.0 - torch.arange(n_bins + 1, device=r.device, dtype=torch.float64) / n_bins)
    f[-1] = 1.0
    e = r_out[:, None] * f[None, :]
    lo = st[:, None].expand(nh, n_bins + 1).clone()
    hi = (st + cnt)[:, None].expand(nh, n_bins + 1).clone()
    while bool((lo < hi).any()):                    # first position with r > e
        mid = (lo + hi) // 2
        le = r[mid.clamp(max=r.shape[0] - 1)] <= e
        go = lo < hi
        lo = torch.where(go & le, mid + 1, lo)
        hi = torch.where(go & ~le, mid, hi)
    inner = mi[lo] - mi[st][:, None]
    out = torch.zeros(nh, n_bins, 4, dtype=torch.float64, device=r.device)
    out[:, :, 0] = (lo[:, 1:] - lo[:, :-1]).double()
    out[:, :, 1] = inner[:, 1:]
    out[:, :, 2] = (inner[:, 1:] - inner[:, :-1]) / (4.0 * math.pi / 3.0 * (e[:, 1:] ** 3 - e[:, :-1] ** 3))
    out[:, :, 3] = (prm.G * inner[:, 1:] / e[:, 1:]).sqrt()
    return torch.where((cnt > 0)[:, None, None], out, torch.zeros_like(out))


def _props(h, off, vel, m, phi, cnt, k_vir, prm):
    """The fields of ahf_halo_properties from the bound sets' FP64 offsets."""
    nh, dev = cnt.shape[0], m.device
    st = _starts(cnt)
    pos = torch.arange(m.shape[0], device=dev) - st[h]
    n_use = torch.where(k_vir >= 0, k_vir + 1, cnt)
    use = pos < n_use[h]
    h, m, phi = h[use], m[use], phi[use]
    off, vel = [x[use] for x in off], [x[use] for x in vel]
    st = _starts(n_use)

    def total(x):
        return _seg_cum(x, st, n_use)[1]

    M = total(m)
    vb = [total(m * v) / M for v in vel]
    u = [vel[a] - vb[a][h] + prm.H * off[a] for a in range(3)]
    J = [total(m * (off[(a + 1) % 3] * u[(a + 2) % 3] - off[(a + 2) % 3] * u[(a + 1) % 3])) for a in range(3)]
    K = 0.5 * total(m * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
    U = 0.5 * total(m * phi)
    E = K + U
    lam = (J[0] ** 2 + J[1] ** 2 + J[2] ** 2).sqrt() * E.abs().sqrt() / (prm.G * M * M * M.sqrt())
    r = (off[0] ** 2 + off[1] ** 2 + off[2] ** 2).sqrt()
    q = torch.where(r > 0, _seg_cum(m, st, n_use)[0] / r, torch.zeros_like(r))
    best = torch.zeros(nh, dtype=torch.float64, device=dev).scatter_reduce(0, h, q, "amax")
    is_best = q == best[h]
    rmax = torch.full((nh,), math.inf, dtype=torch.float64, device=dev)
    rmax = rmax.scatter_reduce(0, h[is_best], r[is_best], "amin")
    out = torch.stack([n_use.double(), M, *J, K, U, E, lam, (prm.G * best).sqrt(), rmax, (k_vir >= 0).double()], 1)
    return torch.where((n_use > 0)[:, None], out, torch.cat([torch.zeros_like(out[:, :11]), out[:, 11:]], 1))


def exact(case, seed):
    n_most = case["haloes"] * case["hi"]
    if case["coord"] == "box" and n_most > EXACT_MAX:
        return None
    parts, halos, subs = _population(case, seed)
    prm = _params(case)
    kind = case["kind"]
    members, parent = None, None
    if kind == "hierarchy":
        halos, parent, members = _hierarchy(parts, halos, subs)
    dev = parts.x.device
    nh = len(halos)
    count = torch.from_numpy(halos["count"].copy()).to(dev)
    hid = torch.repeat_interleave(torch.arange(nh, device=dev), count)
    idx = torch.arange(parts.n, device=dev) if members is None else members
    off = []
    for x, name in zip((parts.x, parts.y, parts.z), ("cx", "cy", "cz")):
        d = x[idx].double() - torch.from_numpy(halos[name].copy()).to(dev)[hid]
        if prm.box > 0:
            d = torch.where(d > 0.5 * prm.box, d - prm.box, d)
            d = torch.where(d < -0.5 * prm.box, d + prm.box, d)
        off.append(d)
    vel = [x[idx].double() for x in (parts.vx, parts.vy, parts.vz)]
    m = parts.m[idx].double() if parts.m is not None else torch.full((idx.shape[0],), parts.m0, dtype=torch.float64,
                                                                     device=dev)
    u_th = None if parts.u_th is None else parts.u_th[idx].double()
    radius = torch.from_numpy(halos["radius"].copy()).to(dev)
    if parent is None:
        got = _unbind(off, vel, m, u_th, hid, nh, radius, prm)
    else:
        # subhaloes first, then each host without what its subhaloes bound
        is_sub = torch.from_numpy(parent >= 0).to(dev)
        a = _unbind(off, vel, m, u_th, hid, nh, radius, prm, is_sub[hid])
        owned = torch.zeros(parts.n, dtype=torch.bool, device=dev)
        owned[idx[a[0]]] = True
        b = _unbind(off, vel, m, u_th, hid, nh, radius, prm, ~is_sub[hid] & ~owned[idx])
        got = [torch.cat([x, y]) for x, y in zip(b[:5], a[:5])]
        got += [a[5] + b[5], a[6] + b[6]]
    slot, h, r, mb, phi, cnt, vb = got
    mv, rv, kv = _virial(h, r, mb, cnt, prm)
    rec = {"ids": None, "m_vir": mv, "r_vir": rv, "vbulk": vb}
    if kind == "serve":
        return {**{k: None if x is None else x.cpu() for k, x in rec.items()}, "bound": None}
    if kind == "catalogue":
        props = _props(h, [x[slot] for x in off], [x[slot] for x in vel], mb, phi, cnt, kv, prm)
        # the second catalogue's halo k holds the particles from the first
        # quarter of its slots on
        inside = slot - torch.from_numpy(halos["offset"].copy()).to(dev)[h] >= (count // 4)[h]
        shared = torch.bincount(h[inside], minlength=nh).double()
        nb = (count - count // 4).double()
        xi = torch.where(cnt > 0, shared * shared / (cnt.double() * nb), torch.zeros_like(nb))
        rows = _rows(h, r, mb, cnt, rv, case["bins"], prm)
        return {"prof": _columns(rows, 4), "props": _columns(props, ahf.PROP_FIELDS), "best": None, "shared": None,
                "xi": xi}
    out_phi = torch.zeros(idx.shape[0], dtype=torch.float64, device=dev)
    st = _starts(cnt)
    where = torch.from_numpy(halos["offset"].copy()).to(dev)[h] + torch.arange(h.shape[0], device=dev) - st[h]
    out_phi[where] = phi
    res = {**rec, "bound": None, "phi": out_phi, "removed": None}
    if kind in ("unbind_profile", "host"):
        res["prof"] = _columns(_rows(h, r, mb, cnt, rv, case["bins"], prm), 4)
    return res
