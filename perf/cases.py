"""The work that a user of this library has it do, as measured cases.

Every case is a block of Monte Carlo sweeps through the public entry points
(a temperature point: reset the averages, equilibrate, measure, read the
averages and the spins), a batch of such points as one group, a call on
caller-owned device spins, or a set of jobs through the server.  Sizes are
those of the repository's own workloads, tests and studies.

A case is a dict of plain values:
  kind        "lattice", "group", "noalloc" or "serve"
  lx, ly, lz  sites (cells of a crystal); "sizes" for the cubes of a group or
              of the jobs, cycled over "count" lattices
  precision   "f32" or "f64"
  faces       one letter per axis: p periodic, o open, k pinned, a anti-periodic
  crystal     "sc", "bcc", "fcc" or "hcp"; j2 next-nearest exchange
  ku, kc, hz  uniaxial and cubic anisotropy, field along z; t temperature
  torque      whether samples hold the torques
  grain       mean grain diameter of a Voronoi film (0: no film)
  wall        whether the start is a domain wall along x
  profile     slice profile every so many measured sweeps (0: none)
  theta, phi  direction of a constrained run (theta < 0: unconstrained)
  eq, meas    unmeasured, then measured sweeps
"""
import math
import time

import numpy as np
import torch

import paper_2103_03517_gb300 as mc

_PLAIN = dict(kind="lattice", precision="f32", faces="ppp", crystal="sc", j2=0.0, ku=0.01, kc=0.0, hz=0.0, t=0.8,
              torque=True, grain=0.0, wall=False, profile=0, theta=-1.0, phi=0.0, eq=0, meas=0)
_FACE = {"p": mc.MC_PERIODIC, "o": mc.MC_OPEN, "k": mc.MC_PINNED, "a": mc.MC_ANTIPERIODIC}
_CRYSTAL = {"sc": mc.MC_SC, "bcc": mc.MC_BCC, "fcc": mc.MC_FCC, "hcp": mc.MC_HCP}
_NSUB = {"sc": 1, "bcc": 2, "fcc": 4, "hcp": 4}


def _case(name=None, **kw):
    c = dict(_PLAIN, **kw)
    if name is not None:
        c["name"] = name
    return c


def _cube(n):
    return dict(lx=n, ly=n, lz=n)


def listed():
    return [
        # the reference point: 16^3 in double precision, the mode that reproduces a serial run bit for bit
        _case("point_16_f64", **_cube(16), precision="f64", t=0.5, eq=100, meas=100),
        # the first thing a new user runs: one 64^3 lattice below T_C
        _case("cube_64", **_cube(64), eq=100, meas=100),
        # the headline lattice alone
        _case("cube_128", **_cube(128), eq=100, meas=100, torque=False),
        # a magnetisation curve: 32 lattices of uneven size and temperature advanced together
        _case("batch_mt_32", kind="group", sizes="16 32 64 128", count=32, t=0.05, eq=20, meas=20),
        # the mesh of the published stiffness study, a size that is no power of two
        _case("cube_160", **_cube(160), ku=0.042, t=0.6, eq=20, meas=20),
        # a free-standing particle: odd ragged sizes, open faces, cubic anisotropy, a field
        _case("particle_open", lx=90, ly=75, lz=61, faces="ooo", ku=0.0, kc=0.05, hz=0.1, t=0.7, eq=40, meas=40),
        # the Bloch wall between pinned end planes, its profile averaged on the way
        _case("wall_1024", lx=1024, ly=128, lz=128, faces="kpp", ku=0.05, t=0.6, wall=True, profile=10, torque=False,
              eq=10, meas=20),
        # a granular recording film: bond mask, an easy axis per grain, grain magnetisations
        _case("film_1024", lx=1024, ly=1024, lz=15, faces="ppo", ku=0.02, t=0.9, grain=10.0, eq=10, meas=10),
        # a real crystal structure
        _case("fcc_96", **_cube(96), crystal="fcc", ku=0.02, t=1.5, eq=10, meas=10),
        # the anisotropy study: constrained runs over direction and temperature as one group
        _case("constrained_64_x80", kind="group", sizes="64", count=80, ku=0.05, kc=0.02, t=0.2, theta=0.0, eq=10,
              meas=10),
        # a few sweeps inside another program's loop, on device memory that the caller owns
        _case("noalloc_64", kind="noalloc", **_cube(64), ku=0.01, t=0.8, meas=4),
        # a mix of small temperature and constrained jobs through the server
        _case("serve_24", kind="serve", sizes="8 16 32 64", count=24, ku=0.02, t=0.6, eq=50, meas=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return max(2, n - n % 2)


def draw(rng):
    kind = rng.choice(["cube", "cube", "box", "open", "wall", "film", "crystal", "f64", "constrained", "group", "noalloc",
                       "serve"])
    t = round(rng.uniform(0.1, 1.5), 3)
    ku = round(rng.choice([0.0, rng.uniform(0.005, 0.05)]), 4)
    kc = round(rng.choice([0.0, 0.0, rng.uniform(0.01, 0.05)]), 4)
    torque = rng.random() < 0.6
    budget = 2e8  # updates of a pass

    def sweeps(n, most=200, budget=budget):
        s = max(2, min(most, int(budget / n)))
        return rng.randint(max(1, s // 2), s)

    if kind == "cube":
        L = _even(_log_int(rng, 8, 256))
        e = sweeps(L ** 3)
        return _case(**_cube(L), t=t, ku=ku, kc=kc, torque=torque, eq=e, meas=e)
    if kind == "box":
        d = dict(lx=_even(_log_int(rng, 16, 256)), ly=_even(_log_int(rng, 8, 200)), lz=_even(_log_int(rng, 4, 200)))
        e = sweeps(d["lx"] * d["ly"] * d["lz"])
        return _case(**d, t=t, ku=ku, kc=kc, hz=round(rng.choice([0.0, rng.uniform(0.0, 0.3)]), 3), torque=torque, eq=e,
                     meas=e)
    if kind == "open":
        d = dict(lx=_even(_log_int(rng, 10, 200)), ly=_log_int(rng, 7, 150), lz=_log_int(rng, 3, 150))
        e = sweeps(d["lx"] * d["ly"] * d["lz"], 100)
        return _case(**d, faces="ooo", t=t, ku=ku, kc=kc, hz=0.1, torque=torque, eq=e, meas=e)
    if kind == "wall":
        yz = _even(_log_int(rng, 16, 128))
        lx = rng.choice([128, 256, 384, 512, 768, 1024, 200, 334])
        e = sweeps(lx * yz * yz, 60)
        return _case(lx=lx, ly=yz, lz=yz, faces=rng.choice(["kpp", "app"]), ku=round(rng.uniform(0.008, 0.05), 4),
                     t=round(rng.uniform(0.1, 1.1), 3), wall=True, profile=10, torque=False, eq=e, meas=max(10, e - e % 10))
    if kind == "film":
        xy = rng.choice([128, 192, 256, 384, 512, 768])
        d = dict(lx=xy, ly=xy, lz=rng.randint(2, 24))
        e = sweeps(xy * xy * d["lz"], 40)
        return _case(**d, faces="ppo", ku=0.02, t=t, grain=round(rng.uniform(8.0, 64.0), 1), eq=e, meas=e)
    if kind == "crystal":
        c = rng.choice(["bcc", "fcc", "hcp"])
        L = _even(_log_int(rng, 8, 96))
        e = sweeps(_NSUB[c] * L ** 3, 60, budget / 2)
        return _case(**_cube(L), crystal=c, j2=round(rng.choice([0.0, 0.2]), 2) if c != "hcp" else 0.0,
                     ku=round(rng.uniform(0.0, 0.05), 4), t=round(rng.uniform(0.2, 2.5), 3), torque=torque, eq=e, meas=e)
    if kind == "f64":
        d = dict(lx=_even(_log_int(rng, 8, 64)), ly=_even(_log_int(rng, 8, 64)), lz=_even(_log_int(rng, 8, 64)))
        e = sweeps(d["lx"] * d["ly"] * d["lz"], 100, 4e6)
        return _case(**d, precision="f64", t=t, ku=ku, kc=kc, eq=e, meas=e)
    if kind == "constrained":
        L = _even(_log_int(rng, 8, 256))
        e = sweeps(L ** 3, 60, budget / 2)
        return _case(**_cube(L), t=round(rng.uniform(0.1, 1.2), 3), ku=0.05, kc=kc, theta=float(rng.randrange(0, 91, 10)),
                     phi=rng.choice([0.0, 45.0]), eq=e, meas=e)
    if kind == "group":
        sizes = rng.choice(["16 32 64 128", "16", "32", "64", "48 96", "24 40 56", "128", "8 16 32"])
        count = _log_int(rng, 2, 64)
        n = sum(int(sizes.split()[i % len(sizes.split())]) ** 3 for i in range(count))
        con = rng.random() < 0.4
        e = sweeps(n, 60, budget / 2)
        return _case(kind="group", sizes=sizes, count=count, ku=0.05 if con else 0.01, kc=0.02 if con else 0.0,
                     t=0.2 if con else 0.05, theta=0.0 if con else -1.0, torque=torque, eq=e, meas=e)
    if kind == "noalloc":
        L = _even(_log_int(rng, 8, 128))
        return _case(kind="noalloc", **_cube(L), ku=ku, t=t, meas=rng.randint(1, 8))
    return _case(kind="serve", sizes=rng.choice(["8 16 32 64", "16 32", "8", "32 64 12 20"]), count=_log_int(rng, 4, 32),
                 ku=0.02, t=0.6, eq=rng.randint(20, 80), meas=rng.randint(20, 160))


# ------------------------------------------------------------------ inputs
def _cubes(case):
    sizes = [int(s) for s in case["sizes"].split()]
    return [sizes[i % len(sizes)] for i in range(case["count"])]


def _direction(theta, phi):
    a, b = math.radians(theta), math.radians(phi)
    return (math.sin(a) * math.cos(b), math.sin(a) * math.sin(b), math.cos(a))


def _start(dims, nsub, t, seed, f64=False, direction=(0.0, 0.0, 1.0), wall=False):
    """Spins near equilibrium at temperature t in the device layout (2 nsub
    colour arrays of 3 components, each padded to a multiple of 64 with
    zeros): the direction, or a wall along x, with a random tilt."""
    lx, ly, lz = dims
    nc = lx * ly * lz // 2
    stride = (nc + 63) // 64 * 64
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn((2 * nsub, 3, stride), generator=g, device="cuda", dtype=torch.float32)
    v *= 0.45 * math.sqrt(t)
    if wall:  # rotates from +z to -z in the y-z plane, end planes exactly on the axis
        q = torch.arange(nc, device="cuda")
        row = q // (lx // 2)
        for c in range(2):
            x = 2 * (q % (lx // 2)) + (row % ly + row // ly + c) % 2
            a = math.pi / (1.0 + torch.exp(-(x - (lx - 1) / 2.0) / 4.5))
            v[c, 1, :nc] += torch.sin(a)
            v[c, 2, :nc] += torch.cos(a)
            for end, s in ((0, 1.0), (lx - 1, -1.0)):
                v[c, 0, :nc][x == end] = 0.0
                v[c, 1, :nc][x == end] = 0.0
                v[c, 2, :nc][x == end] = s
    else:
        v += torch.tensor(direction, device="cuda", dtype=torch.float32)[None, :, None]
    v = v.double()
    v /= v.norm(dim=1, keepdim=True)
    v[:, :, nc:] = 0.0
    return v.reshape(-1) if f64 else v.float().reshape(-1)


def _voronoi(lx, ly, lz, diameter, seed):
    """Columnar grains of an lx x ly x lz film, periodic in the plane: one
    grain centre per cell of a jittered grid, each column owned by the
    nearest.  Returns grain ids and bond bits per site and the easy axes."""
    cell = diameter * math.sqrt(math.pi) / 2.0
    nx, ny = max(3, int(lx / cell)), max(3, int(ly / cell))
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((ny, nx, 2), generator=g, device="cuda", dtype=torch.float64)
    axes = torch.randn((ny * nx, 3), generator=g, device="cuda", dtype=torch.float64)
    axes /= axes.norm(dim=1, keepdim=True)
    cx, cy = lx / nx, ly / ny
    x = torch.arange(lx, device="cuda", dtype=torch.float64)[None, :] + 0.5
    y = torch.arange(ly, device="cuda", dtype=torch.float64)[:, None] + 0.5
    best = torch.full((ly, lx), 1e30, device="cuda", dtype=torch.float64)
    owner = torch.zeros((ly, lx), device="cuda", dtype=torch.int32)
    for dj in (-2, -1, 0, 1, 2):
        for di in (-2, -1, 0, 1, 2):
            i, j = torch.floor(x / cx).long() + di, torch.floor(y / cy).long() + dj
            p = u[(j % ny).expand(ly, lx), (i % nx).expand(ly, lx)]
            d = ((i + p[..., 0]) * cx - x) ** 2 + ((j + p[..., 1]) * cy - y) ** 2
            near = d < best
            best = torch.where(near, d, best)
            owner = torch.where(near, ((j % ny) * nx + i % nx).int(), owner)
    bits = torch.zeros((ly, lx), device="cuda", dtype=torch.uint8)
    for b, (shift, dim) in enumerate(((1, 1), (-1, 1), (1, 0), (-1, 0))):
        bits |= (owner == torch.roll(owner, shift, dim)).to(torch.uint8) << b
    mask = bits[None].repeat(lz, 1, 1)
    mask[1:] |= 16
    mask[:-1] |= 32
    gid = owner[None].expand(lz, ly, lx).contiguous()
    return gid.reshape(-1).cpu().numpy(), mask.reshape(-1).cpu().numpy(), axes.cpu().numpy()


def _seed64(seed, i=0):
    return (int(seed) * 1000003 + 7919 * i + 17) % (1 << 63)


def _desc(case, dims, seed, t, **more):
    return mc.make_desc(dims, J=1.0, K_u=case["ku"], K_c=case["kc"], H=(0.0, 0.0, case["hz"]), T=t, seed=seed,
                        precision=mc.MC_FP64 if case["precision"] == "f64" else mc.MC_FP32,
                        boundary=tuple(_FACE[f] for f in case["faces"]), lattice=_CRYSTAL[case["crystal"]], J2=case["j2"],
                        sample_torque=case["torque"], ring_capacity=256, **more)


class _Program:
    """What a user's program keeps between calls: handles, and pinned host
    memory for the spins that it reads back."""

    def __init__(self, case):
        self.case = case
        self.handles, self.group, self.server = [], None, None
        self.spins = []

    def lattice(self, desc, start):
        h = mc.mc_create_ex(desc)
        self.handles.append(h)
        host = torch.empty(start.shape, dtype=start.dtype, pin_memory=True)
        host.copy_(start)
        mc.mc_import_state(h, host.data_ptr(), mc.mc_state_bytes(h))
        mc.mc_sync(h)
        self.spins.append(host)

    def __del__(self):
        if self.server is not None:
            mc.mc_server_destroy(self.server)
        if self.group is not None:
            mc.mc_group_destroy(self.group)
        for h in self.handles:
            mc.mc_destroy(h)


def _jobs(case, seed):
    """(desc arguments, kind, theta) of the server's jobs: temperature points
    and constrained points in turn."""
    rng = np.random.default_rng(seed)
    for i, L in enumerate(_cubes(case)):
        yield L, round(float(rng.uniform(0.05, 1.2)), 3), i % 2 == 1, float(rng.integers(0, 10) * 10), _seed64(seed, i)


def _points(case):
    """(T, theta, phi) of the lattices of a group: a temperature sweep, or a
    sweep of directions at four temperatures."""
    out = []
    for i in range(case["count"]):
        if case["theta"] < 0:
            out.append((case["t"] * (i + 1) if case["t"] * case["count"] <= 1.7 else 0.05 + 1.5 * i / case["count"], 0.0,
                        0.0))
        else:
            out.append(((0.2, 0.6, 1.0, 1.3)[i * 4 // case["count"]], float(i % 10 * 10), 45.0 * (i // 10 % 2)))
    return out


def prepare(case, seed):
    s = _Program(case)
    kind = case["kind"]
    if kind == "noalloc":
        dims = (case["lx"], case["ly"], case["lz"])
        s.dims, s.seed, s.theta, s.first = dims, _seed64(seed), 30, 0
        s.dev = _start(dims, 1, case["t"], seed)
        s.samples = torch.zeros((case["meas"], 14), device="cuda", dtype=torch.float64)
        torch.cuda.synchronize()
        return s
    if kind == "serve":
        s.server = mc.mc_server_create()
        s.jobs = []
        for L, t, con, theta, sd in _jobs(case, seed):
            d = mc.make_desc((L, L, L), K_u=case["ku"], T=t, seed=sd, init_dir=_direction(theta, 0.0) if con else (0, 0, 1))
            s.jobs.append(mc.make_job(d, mc.MC_JOB_CONSTRAINED if con else mc.MC_JOB_SWEEP, theta_c_deg=theta,
                                      n_equilibrate=case["eq"], n_measure=case["meas"]))
        return s
    if kind == "group":
        pts = _points(case)
        for i, L in enumerate(_cubes(case)):
            t, th, ph = pts[i]
            con = case["theta"] >= 0
            s.lattice(_desc(case, (L, L, L), _seed64(seed, i), t),
                      _start((L, L, L), 1, t, seed * 131 + i, direction=_direction(th, ph) if con else (0.0, 0.0, 1.0)))
        s.group = mc.mc_group_create(s.handles)
        s.th = np.array([p[1] for p in pts])
        s.ph = np.array([p[2] for p in pts])
        return s
    dims = (case["lx"], case["ly"], case["lz"])
    more = {}
    if case["grain"] > 0:
        gid, mask, axes = _voronoi(*dims, case["grain"], seed)
        more = dict(grain_id=gid, bond_mask=mask, grain_axis=axes)
        s.n_grains = len(axes)
    if case["wall"]:
        more["init"] = mc.MC_INIT_WALL
    direction = _direction(case["theta"], case["phi"]) if case["theta"] >= 0 else (0.0, 0.0, 1.0)
    s.lattice(_desc(case, dims, _seed64(seed), case["t"], **more),
              _start(dims, _NSUB[case["crystal"]], case["t"], seed, case["precision"] == "f64", direction, case["wall"]))
    return s


# --------------------------------------------------------------------- run
def _read(o):
    """The averages of one lattice: whole numbers, then the doubles."""
    return [o.n_samples, o.sweeps_done, o.theta_deg, o.error], np.frombuffer(o, np.float64, offset=24)


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "noalloc":
        s.theta = mc.mc_sweep_noalloc(s.dev.data_ptr(), s.dims, 1.0, case["ku"], (0, 0, 1), case["kc"],
                                      (0, 0, case["hz"]), case["t"], s.seed, s.first, case["meas"], s.theta,
                                      s.samples.data_ptr(), torch.cuda.current_stream().cuda_stream)
        s.first += case["meas"]
        return {"theta": s.theta, "spins": s.dev, "samples": s.samples}
    if kind == "serve":
        ids = [mc.mc_submit(s.server, j) for j in s.jobs]
        results = {}
        while len(results) < len(ids):
            for i in ids:
                if i not in results:
                    rc, r = mc.mc_poll(s.server, i)
                    if rc == mc.MC_OK:
                        results[i] = r
                        mc.mc_forget(s.server, i)
            time.sleep(1e-4)
        both = [_read(results[i].obs) for i in ids]
        return {"status": np.array([results[i].status for i in ids]), "counts": np.array([b[0] for b in both]),
                "averages": np.stack([b[1] for b in both])}
    for h in s.handles:
        mc.mc_reset_stats(h)
    if kind == "group":
        if case["theta"] >= 0:
            mc.mc_group_constrained_sweep(s.group, s.th, s.ph, case["eq"])
            mc.mc_group_constrained_sweep(s.group, s.th, s.ph, case["meas"], True)
        else:
            mc.mc_group_sweep(s.group, case["eq"])
            mc.mc_group_sweep(s.group, case["meas"], True)
        both = [_read(o) for o in mc.mc_group_measure(s.group, len(s.handles))]
        return {"counts": np.array([b[0] for b in both]), "averages": np.stack([b[1] for b in both])}
    h, = s.handles
    out = {}
    if case["theta"] >= 0:
        mc.mc_constrained_sweep(h, case["theta"], case["phi"], case["eq"])
        mc.mc_constrained_sweep(h, case["theta"], case["phi"], case["meas"], True)
    else:
        mc.mc_sweep(h, case["eq"])
        if case["profile"]:
            for _ in range(case["meas"] // case["profile"]):
                mc.mc_sweep(h, case["profile"], True)
                mc.mc_profile_sample(h)
        else:
            mc.mc_sweep(h, case["meas"], True)
    if case["grain"] > 0:
        mc.mc_grain_sample(h)
    out["counts"], out["averages"] = _read(mc.mc_measure(h))
    if case["profile"]:
        out["profile"] = [mc.mc_profile(h, a, case["lx"]) for a in range(3)]
    if case["grain"] > 0:
        out["grains"] = mc.mc_grain_magnetization(h, s.n_grains)[0]
    mc.mc_export_state(h, s.spins[0].data_ptr(), mc.mc_state_bytes(h))
    out["spins"] = s.spins[0]
    return out


def work(case):
    """Every sweep of a lattice reads and writes each spin once (the cone
    angle of a sweep needs the count of the whole sweep before it, so sweeps
    do not fuse): 24 bytes an update in single, 48 in double precision.  An
    update is about 120 operations: six neighbours summed (18), the trial
    point on the cone (45), the energy change (35), the test, the sample."""
    kind = case["kind"]
    if kind in ("group", "serve"):
        n = sum(L ** 3 for L in _cubes(case))
    else:
        n = _NSUB[case["crystal"]] * case["lx"] * case["ly"] * case["lz"]
    updates = n * (case["eq"] + case["meas"])
    return {"bytes": updates * (48 if case["precision"] == "f64" else 24), "flops": updates * 120}


# ------------------------------------------------------------------- exact
def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 of the counters (arrays or numbers), as four uint64 arrays."""
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    m = np.uint64(0xFFFFFFFF)
    x = [np.broadcast_to(np.asarray(v, np.uint64), c0.shape).copy() for v in (c0, c1, c2, c3)]
    for _ in range(10):
        p0, p1 = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        s = np.uint64(32)
        x = [(p1 >> s) ^ x[1] ^ np.uint64(k0), p1 & m, (p0 >> s) ^ x[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x


def _trial_f64(S, c, site, sweep, colour, key):
    """Double precision: a point of the disk by rejection, mapped to the cap
    about S in the frame of Duff et al. (2017)."""
    w = _philox(site, sweep, colour, 0, key)
    P = w[2] * 2.0 ** -32
    u, v = w[0] * 2.0 ** -31 - 1.0, w[1] * 2.0 ** -31 - 1.0
    s = u * u + v * v
    for attempt in range(1, 16):
        bad = np.flatnonzero(~(s < 1.0))
        if not len(bad):
            break
        w = _philox(site[bad], sweep, colour, attempt, key)
        u[bad], v[bad] = w[0] * 2.0 ** -31 - 1.0, w[1] * 2.0 ** -31 - 1.0
        s[bad] = u[bad] * u[bad] + v[bad] * v[bad]
    sc = s * c
    zp, r = 1.0 - sc, np.sqrt(np.maximum(c * (2.0 - sc), 0.0))
    x, y, z = S.T
    g = np.copysign(1.0, z)
    a = -1.0 / (g + z)
    b = x * y * a
    n = ((u * r) * np.stack([1.0 + g * x * x * a, g * b, -g * x]) + (v * r) * np.stack([b, g + y * y * a, -y]) + zp * S.T).T
    return n / np.linalg.norm(n, axis=1, keepdims=True), P, s < 1.0


def _trial_f32(S, c, site, second, sweep, colour, key):
    """Single precision's law in 64 bits: one counter per two neighbouring
    sites of a colour (second: the other site of the two), the cap drawn
    directly and carried onto S by a reflection."""
    w = _philox(site, sweep, colour, 0, key)
    a, b = np.where(second, w[1], w[0]).astype(np.int64), np.where(second, w[3], w[2]).astype(np.int64)
    P = (a >> 10) * 2.0 ** -22
    s = (((a & 0x3FF) << 11) | (b & 0x7FF)) * 2.0 ** -21
    phi = ((b >> 11) * 2.0 ** -21 - 0.5) * (2.0 * math.pi)
    sc = s * c
    r = np.sqrt(sc * (2.0 - sc))
    g = np.copysign(1.0, S[:, 2])
    p = np.stack([r * np.cos(phi), r * np.sin(phi), -g * (1.0 - sc)], 1)
    v = S + np.stack([0.0 * g, 0.0 * g, g], 1)
    n = p - ((v * p).sum(1) / (1.0 + g * S[:, 2]))[:, None] * v
    return n / np.linalg.norm(n, axis=1, keepdims=True), P


def _cubic(S):
    x, y, z = (S * S).T
    return x * y + x * z + y * z


def _chain(case, dims, start, key, sweeps, measured_from, theta=30):
    """The sweeps of a simple cubic lattice without film tables in 64 bits:
    spins in the device layout, theta, and per measured sweep the row
    (sweep, theta, accepted, m, energies, torque, 0)."""
    lx, ly, lz = dims
    nc = lx * ly * lz // 2
    f64 = case["precision"] == "f64"
    dev = start.double().cpu().numpy().reshape(2, 3, -1).copy()
    q = np.arange(nc)
    row = q // (lx // 2)
    at, wrap = [], []  # site of every colour index
    for c in range(2):
        at.append((2 * (q % (lx // 2)) + (row % ly + row // ly + c) % 2) + lx * row)
    S = np.zeros((lx * ly * lz, 3))
    for c in range(2):
        S[at[c]] = dev[c, :, :nc].T
    x, y, z = np.arange(lx * ly * lz) % lx, np.arange(lx * ly * lz) // lx % ly, np.arange(lx * ly * lz) // (lx * ly)
    nb, fac = [], []
    pin = np.zeros(lx * ly * lz, bool)
    for pos, L, unit, f in ((x, lx, 1, case["faces"][0]), (y, ly, lx, case["faces"][1]), (z, lz, lx * ly, case["faces"][2])):
        w = {"p": 1.0, "a": -1.0, "o": 0.0, "k": 0.0}[f]
        for step in (-1, 1):
            other = (pos + step) % L
            nb.append(np.arange(lx * ly * lz) + (other - pos) * unit)
            fac.append(np.where(np.abs(other - pos) != 1, w, 1.0) if L > 2 else
                       np.where((pos + step < 0) | (pos + step >= L), w, 1.0))
        if f == "k":
            pin |= (pos == 0) | (pos == L - 1)
    n_mov = int((~pin).sum())
    ku, kc, hz, t = case["ku"], case["kc"], case["hz"], case["t"]
    rows = []
    n = float(len(S))
    for sweep in range(sweeps):
        cone = 2.0 * math.sin(math.radians(theta) / 2.0) ** 2
        acc = 0
        for c in range(2):
            i = at[c]
            h = np.zeros((nc, 3))
            for d in range(6):
                h = h + fac[d][i, None] * S[nb[d][i]]
            old = S[i]
            if f64:
                new, P, ok = _trial_f64(old, cone, i.astype(np.uint64), sweep, c, key)
            else:
                new, P = _trial_f32(old, cone, i[q & ~1].astype(np.uint64), (q & 1) == 1, sweep, c, key)
                ok = True
            d = new - old
            dE = (-(d * h).sum(1) - ku * (new[:, 2] ** 2 - old[:, 2] ** 2) + kc * (_cubic(new) - _cubic(old)) - hz * d[:, 2])
            take = ok & ~pin[i] & ((dE <= 0.0) | (P < np.exp(np.minimum(-dE / t, 0.0))))
            S[i] = np.where(take[:, None], new, old)
            acc += int(take.sum())
        theta = min(theta + 1, 180) if 2 * acc > n_mov else max(theta - 1, 1)
        if sweep >= measured_from:
            m = S.mean(0)
            ex = sum((fac[d][at[1], None] * S[nb[d][at[1]]] * S[at[1]]).sum() for d in range(6))
            sx, sy, sz = S.T
            x2, y2, z2 = (S * S).T
            g = np.stack([sx * (y2 + z2), sy * (x2 + z2), sz * (x2 + y2)], 1)
            zero = 0.0 * sz
            tau = (2.0 * ku * np.stack([sz * sy, -sz * sx, zero], 1) - 2.0 * kc * np.cross(S, g)
                   + hz * np.stack([sy, -sx, zero], 1)).sum(0) / n
            parts = [-ex / n, -ku * (sz * sz).sum() / n, kc * _cubic(S).sum() / n, -hz * m[2]]
            rows.append([sweep, theta, acc, *m, *parts, *(tau if case["torque"] else 0.0 * tau), 0.0])
    for c in range(2):
        dev[c, :, :nc] = S[at[c]].T
    return dev.reshape(-1), theta, np.array(rows), acc / n_mov


def exact(case, seed):
    """In 64 bits a chain is determined by its draws for as long as rounding
    flips no acceptance: over hundreds of sweeps of a small lattice in double
    precision, over a few sweeps in single.  A longer single-precision chain
    parts from the 64-bit one at its first flipped move and is then another
    sample of the same ensemble, so it has no such value."""
    dims = (case.get("lx", 0), case.get("ly", 0), case.get("lz", 0))
    if case["kind"] == "noalloc":
        if dims[0] * dims[1] * dims[2] * case["meas"] > 2e7:
            return None
        spins, theta, rows, _ = _chain(case, dims, _start(dims, 1, case["t"], seed), _seed64(seed), case["meas"], 0)
        return {"theta": None, "spins": spins, "samples": rows}
    if case["kind"] != "lattice" or case["precision"] != "f64" or case["theta"] >= 0 or case["crystal"] != "sc":
        return None
    spins, theta, rows, acc = _chain(case, dims, _start(dims, 1, case["t"], seed, True), _seed64(seed),
                                     case["eq"] + case["meas"], case["eq"])
    m, parts, tau = rows[:, 3:6], rows[:, 6:10], rows[:, 10:13]
    ml, e = np.linalg.norm(m, axis=1), parts.sum(1)
    nt = dims[0] * dims[1] * dims[2] / case["t"]
    chi = [nt * ((ml ** 2).mean() - ml.mean() ** 2), *(nt * ((m ** 2).mean(0) - m.mean(0) ** 2))]
    avg = [acc, *m.mean(0), *(m ** 2).mean(0), *np.abs(m).mean(0), ml.mean(), (ml ** 2).mean(), (ml ** 4).mean(), e.mean(),
           (e ** 2).mean(), *parts.mean(0), *tau.mean(0), *(tau ** 2).mean(0), *chi,
           1.0 - (ml ** 4).mean() / (3.0 * (ml ** 2).mean() ** 2)]
    return {"counts": None, "averages": np.array(avg), "spins": spins}
