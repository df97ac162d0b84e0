"""What a user of this library has it do, as cases that can be timed.

A case is one of five kinds of call sequence, each through the Python binding:

  film      one film: sweeps with records, the final spins (device), the records (host)
  set       a procedure's or a configuration's film set as one batch: sweeps, every film's records
  mixed     a batch of films of unequal sizes, boundaries and temperatures
  serve     jobs submitted to the continuous-batching server, waited for and collected
  snapshot  spins uploaded from device memory, measured, and copied back (checkpoint, resume, analysis)

``work`` counts a spin-flip attempt as 30 integer operations: a Philox4x32-10
call (98 operations) serves four attempts, the neighbour count, the threshold
and the flip take about 5.5 more.  Its bytes are the packed lattice read and
written once per pass, and the outputs.
"""
import numpy as np
import torch

import paper_1411_5588_gb300 as ig
from paper_1411_5588_gb300 import workloads

OPS_PER_ATTEMPT = 30


def _film(name, Lx, Ly, Lz, T, H1, sweeps, every, tune, y=ig.Y_GAPBC, x=ig.X_FREE, H=0.0, init=ig.INIT_SLAB_Y):
    return dict(name=name, kind="film", Lx=Lx, Ly=Ly, Lz=Lz, T=T, H1=H1, H=H, y=y, x=x, init=init, sweeps=sweeps,
                every=every, tune=tune)


def listed():
    return [
        # the 8^3 film of the benchmark's first configuration: a record every sweep, bound by latency
        _film("film_8", 8, 8, 8, 3.0, 0.5, 1000, 1, False, init=ig.INIT_RANDOM),
        # the smallest call in use: ten sweeps of a small film and their one record, read at once
        _film("step_16x48x32", 16, 48, 32, 3.0, 0.5, 10, 10, False),
        # one medium film as a handle gives it without tuning: odd sizes, rows that end in a partial
        # word, a bulk field (every layer has its own thresholds for up and down spins), periodic y
        _film("film_ragged", 37, 75, 214, 2.2, 0.3, 100, 5, False, y=ig.Y_PBC, H=0.05, init=ig.INIT_RANDOM),
        # the benchmark's main film, tuned as the README does, a record every ten sweeps
        _film("film_46m", 120, 240, 1600, 3.0, 0.55, 100, 10, True),
        # that film's state in and out: spins uploaded, measured on demand, copied back
        dict(name="snapshot_46m", kind="snapshot", Lx=120, Ly=240, Lz=1600),
        # the 64-film integration set of the third configuration: four sizes, a record every sweep
        dict(name="ti_64", kind="set", set="ti", sweeps=128, every=1),
        # the contact-angle procedure's 40 films, a record every sweep
        dict(name="contact_angle", kind="set", set="contact_angle", fields=4, nodes=8, sweeps=1000, every=1),
        # the same procedure at one field: ten films, too few to fill the GPU by themselves
        dict(name="one_field", kind="set", set="contact_angle", fields=1, nodes=8, sweeps=1000, every=1),
        # the beta integration's 192 small films of four sizes, energies every ten sweeps
        dict(name="interface_tension", kind="set", set="interface_tension", points=24, sweeps=1000, every=10),
        # the constant-area set of the line tension: thin and thick films of equal area
        dict(name="line_tension", kind="set", set="line_tension", nodes=6, sweeps=500, every=1),
        # jobs of the 2000-job stream's sizes, submitted together
        dict(name="serve_32", kind="serve", jobs=32, mix=3, lo=200, hi=2000, every=10),
        # the temperature scan: forty of the main film
        dict(name="t_scan", kind="set", set="t_scan", sweeps=10, every=1),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _even(v):
    return v + v % 2


def draw(rng):
    kind = rng.choice(["film", "film", "film", "set", "mixed", "mixed", "serve", "snapshot"])
    if kind in ("film", "snapshot"):
        Lx, Ly, Lz = _log(rng, 4, 128), _log(rng, 4, 256), _even(_log(rng, 4, 1600))
        if kind == "snapshot":
            return dict(kind=kind, Lx=Lx, Ly=Ly, Lz=Lz)
        x = ig.X_PBC if Lx % 2 == 0 and rng.random() < 0.15 else ig.X_FREE
        every = rng.choice([0, 1, 1, 2, 5, 10, 10, 20])
        # the paper's range, and now and then a quench to a temperature where some moves never happen
        T = 0.05 if rng.random() < 0.1 else round(rng.uniform(1.5, 4.4), 3)
        sweeps = min(_log(rng, 10, 1000), max(10, int(5e9 / (Lx * Ly * Lz))))
        c = _film("", Lx, Ly, Lz, T, round(rng.uniform(0.0, 1.0), 3), sweeps, every, rng.random() < 0.5,
                  y=rng.choice([ig.Y_GAPBC, ig.Y_GAPBC, ig.Y_PBC, ig.Y_APBC]), x=x,
                  H=rng.choice([0.0, 0.0, 0.0, round(rng.uniform(-0.5, 0.5), 3)]),
                  init=rng.choice([ig.INIT_RANDOM, ig.INIT_SLAB_Y, ig.INIT_ALL_UP]))
        del c["name"]
        return c
    if kind == "set":
        which = rng.choice(["contact_angle", "interface_tension", "line_tension"])
        sweeps, every = rng.randint(200, 600), rng.choice([1, 2, 5, 10])
        if which == "contact_angle":
            return dict(kind=kind, set=which, fields=rng.randint(1, 5), nodes=rng.randint(2, 8), sweeps=sweeps,
                        every=every)
        if which == "interface_tension":
            return dict(kind=kind, set=which, points=rng.randint(2, 24), sweeps=sweeps, every=every)
        return dict(kind=kind, set=which, nodes=rng.randint(1, 6), sweeps=sweeps, every=every)
    if kind == "mixed":
        return dict(kind=kind, films=_log(rng, 2, 64), mix=rng.randrange(1 << 30), top=_log(rng, 32, 256),
                    sweeps=_log(rng, 20, 400), every=rng.choice([0, 1, 1, 3, 10]), tune=rng.random() < 0.5)
    return dict(kind=kind, jobs=_log(rng, 2, 32), mix=rng.randrange(1 << 30), lo=100, hi=_log(rng, 200, 2000), every=10)


def _set_jobs(case, seed):
    which, n = case["set"], case["sweeps"]
    if which == "ti":
        jobs = workloads.ti_batch(n)
    elif which == "t_scan":
        jobs = workloads.t_scan_40(n)
    elif which == "contact_angle":
        H1s = [(0.15, 0.3, 0.45, 0.55, 0.62)[i] for i in range(case["fields"])]
        jobs = workloads.contact_angle_set(H1s=H1s, n_gl=case["nodes"], n_sweeps=n)["jobs"]
    elif which == "interface_tension":
        jobs = workloads.interface_tension_set(n_beta=case["points"], n_sweeps=n)["jobs"]
    else:
        jobs = workloads.line_tension_set(n_gl=case["nodes"], n_sweeps=n)["jobs"]
    return [dict(j, seed=int(j["seed"]) * 1000003 + seed, measure_every=case["every"]) for j in jobs]


def _mixed_jobs(case, seed):
    rng = np.random.RandomState(case["mix"])
    jobs = []
    for i in range(case["films"]):
        Lx, Ly, Lz = (int(round(4.0 * (case["top"] / 4.0) ** u)) for u in rng.random_sample(3))
        jobs.append(dict(Lx=Lx, Ly=Ly, Lz=_even(Lz), T=float(rng.uniform(1.5, 4.4)), H1=float(rng.uniform(0, 1)),
                         y_mode=int(rng.randint(3)), init_kind=int(rng.randint(3)), flip_p=0.01, seed=seed,
                         replica=i, measure_every=case["every"]))
    return jobs


def _serve_jobs(case, seed):
    rng = np.random.RandomState(case["mix"])
    out = []
    for i, j in enumerate(workloads.serve_2000(case["jobs"], seed=case["mix"] % 100003, measure_every=case["every"])):
        out.append(dict(j, seed=seed, replica=i, n_sweeps=int(case["lo"] * (case["hi"] / case["lo"]) ** rng.random_sample())))
    return out


def _jobs(case, seed):
    return {"set": _set_jobs, "mixed": _mixed_jobs, "serve": _serve_jobs}[case["kind"]](case, seed)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind == "film":
        f = ig.Film(case["Lx"], case["Ly"], case["Lz"], J=1.0, H1=case["H1"], T=case["T"], seed=seed, y_mode=case["y"],
                    x_mode=case["x"], H=case["H"])
        f.init(case["init"], 0.01 if case["init"] == ig.INIT_SLAB_Y else 0.0)
        if case["tune"]:
            f.autotune(case["every"])
        if case["every"]:
            f.reserve_records(case["sweeps"] // case["every"] + 1)
        s.update(film=f, spins=torch.empty(f.n_sites, dtype=torch.int8, device="cuda"))
    elif kind == "snapshot":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["Lx"] * case["Ly"] * case["Lz"]
        spins = torch.randint(0, 2, (n,), dtype=torch.int8, device="cuda", generator=g) * 2 - 1
        torch.cuda.synchronize()
        s.update(film=ig.Film(case["Lx"], case["Ly"], case["Lz"], seed=seed), source=spins,
                 spins=torch.empty_like(spins))
    elif kind == "serve":
        s.update(server=ig.Server(1 << 31, 50), jobs=_jobs(case, seed))
    else:
        b = ig.Batch(_jobs(case, seed))
        if kind == "set" or case["tune"]:
            b.autotune()
        if case["every"]:
            b.reserve_records(case["sweeps"] // case["every"] + 1)
        s.update(batch=b, films=len(b))
    return s


def run(state):
    case = state["case"]
    if state["kind"] == "film":
        f = state["film"]
        f.sweep(case["sweeps"], case["every"])
        f.get_spins_device(state["spins"].data_ptr())
        if not case["every"]:
            f.synchronize()
            return {"spins": state["spins"]}
        return {"spins": state["spins"], "records": f.read_series()}
    if state["kind"] == "snapshot":
        f = state["film"]
        f.set_spins_device(state["source"].data_ptr())
        record = f.measure()
        f.get_spins_device(state["spins"].data_ptr())
        f.synchronize()
        return {"record": record, "spins": state["spins"]}
    if state["kind"] == "serve":
        server = state["server"]
        tickets = server.submit(state["jobs"])
        for t in tickets:
            server.wait(t)
        return [server.result(t)[:2] for t in tickets]
    b = state["batch"]
    b.sweep(case["sweeps"], True)
    if not case["every"]:  # without records the spins are what the run was for
        return np.concatenate([b.get_spins(i) for i in range(state["films"])])
    series = [b.read_series(i) for i in range(state["films"])]
    return series if len(series) <= 64 else np.concatenate([r.reshape(-1) for r in series])


def work(case):
    if case["kind"] in ("film", "snapshot"):
        films = [(case["Lx"], case["Ly"], case["Lz"], case.get("sweeps", 0), case.get("every", 0))]
    else:
        films = [(j["Lx"], j["Ly"], j["Lz"], j["n_sweeps"] if case["kind"] == "serve" else case["sweeps"],
                  case["every"]) for j in _jobs(case, 1)]
    b = flops = 0.0
    for Lx, Ly, Lz, sweeps, every in films:
        sites = Lx * Ly * Lz
        flops += OPS_PER_ATTEMPT * sites * sweeps
        b += 2 * sites / 8 + 8.0 * (5 + Lx) * (sweeps // every if every else 0)
        if case["kind"] == "film" or case["kind"] == "serve" or not every:
            b += sites  # the spins as int8
        if case["kind"] == "snapshot":
            b += sites + 8.0 * (5 + Lx)
            flops += 2 * sites
    return {"bytes": b, "flops": flops}


# ------------------------------------------------------------- plain values

_M0, _M1, _W0, _W1, _MASK = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85, 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 over int64 tensors that hold 32-bit words: the four words of each call."""
    for _ in range(10):
        p0, p1 = c0 * _M0, c2 * _M1  # the low 64 bits of the product, whatever its sign
        c0, c1, c2, c3 = ((p1 >> 32) & _MASK) ^ c1 ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ c3 ^ k1, p0 & _MASK
        k0, k1 = (k0 + _W0) & _MASK, (k1 + _W1) & _MASK
    return c0, c1, c2, c3


def _uniform(L, t, key, extra, dev):
    """One 32-bit word per site (Lx, Ly, Lz): word (z0>>1)&3 of the call (row, z0>>3, t, extra | z0&1)."""
    Lx, Ly, Lz = L
    nb = (Lz + 7) // 8
    row = torch.arange(Lx * Ly, device=dev).view(-1, 1, 1).expand(Lx * Ly, nb, 2)
    blk = torch.arange(nb, device=dev).view(1, -1, 1).expand_as(row)
    par = torch.arange(2, device=dev).view(1, 1, 2).expand_as(row)
    words = _philox(row, blk, torch.full_like(row, t), par | extra, *key)
    u = torch.stack(words, 2)  # (row, block, word, parity) is z order inside a block of eight
    return u.reshape(Lx * Ly, nb * 8)[:, :Lz].reshape(Lx, Ly, Lz)


def _neighbours(s, y, x):
    """Sum of the six neighbour spins, and the bond sum, of a film s (Lx, Ly, Lz)."""
    up = s.flip(0) if y == ig.Y_GAPBC else s
    sign = 1 if y == ig.Y_PBC else -1
    yp = torch.cat([s[:, 1:], sign * up[:, :1]], 1)
    ym = torch.cat([sign * up[:, -1:], s[:, :-1]], 1)
    edge = torch.zeros_like(s[:1])
    xp = torch.cat([s[1:], s[:1] if x == ig.X_PBC else edge], 0)
    xm = torch.cat([s[-1:] if x == ig.X_PBC else edge, s[:-1]], 0)
    zp, zm = s.roll(-1, 2), s.roll(1, 2)
    return xp + xm + yp + ym + zp + zm, lambda: int((s * (xp + yp + zp)).sum(dtype=torch.int64))


def _record(s, sweep, y, x):
    m = s.sum((1, 2), dtype=torch.int64)
    return [sweep, _neighbours(s, y, x)[1](), int(m.sum()), int(m[0]), int(m[-1])] + m.tolist()


def _plain_film(L, T, H1, H, y, x, init, p, seed, sweeps, every, dev):
    """The chain and its records from Eq. 1 and the four-phase checkerboard, site by site."""
    Lx, Ly, Lz = L
    key = ((seed & _MASK) ^ (seed >> 32), 0)
    if init == ig.INIT_ALL_UP:
        s = torch.ones(L, dtype=torch.int8, device=dev)
    else:
        u = _uniform(L, _MASK, key, 2, dev)
        if init == ig.INIT_RANDOM:
            up = u < (1 << 31)
        else:
            half = (torch.arange(1, Ly + 1, device=dev) <= Ly // 2).view(1, -1, 1)
            up = half ^ (u < int(np.floor(p * 2.0 ** 32)))
        s = (up.to(torch.int8) * 2 - 1)
    # thresholds by (layer kind, s, sum of neighbours): 2^32 stands for "always"
    kinds = [H + (H1 if k & 1 else 0.0) - (H1 if k & 2 else 0.0) for k in range(4)]
    thr = np.zeros((4, 2, 13), dtype=np.int64)
    for k, h in enumerate(kinds):
        for b, sv in enumerate((-1.0, 1.0)):
            for n in range(-6, 7):
                dE = 2.0 * sv * (float(n) + h)
                thr[k, b, n + 6] = 1 << 32 if dE <= 0.0 else int(np.floor(np.ldexp(np.exp(-dE / T), 32)))
    thr = torch.from_numpy(thr.reshape(-1)).to(dev)
    kind = torch.zeros(Lx, dtype=torch.int64, device=dev)
    kind[0] += 1
    kind[-1] += 2
    colour = (sum(torch.arange(1, n + 1, device=dev).view(*v) for n, v in zip(L, ((-1, 1, 1), (1, -1, 1), (1, 1, -1)))) % 2)
    last = (torch.arange(1, Ly + 1, device=dev) == Ly).view(1, -1, 1)
    records = []
    for t in range(sweeps):
        u = _uniform(L, t, key, 0, dev)
        for c in (0, 1):
            for seam in (False, True):
                nb, _ = _neighbours(s, y, x)
                at = kind.view(-1, 1, 1) * 26 + (s > 0).to(torch.int64) * 13 + nb.to(torch.int64) + 6
                flip = (u < thr[at]) & (colour == c) & (last if seam else ~last)
                s = torch.where(flip, -s, s)
        if every and (t + 1) % every == 0:
            records.append(_record(s, t + 1, y, x))
    out = {"spins": s.reshape(-1).cpu()}
    if every:
        out["records"] = np.array(records, dtype=np.int64).reshape(-1, 5 + Lx)
    return out


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "snapshot":
        g = torch.Generator(device=dev).manual_seed(seed)
        L = (case["Lx"], case["Ly"], case["Lz"])
        s = torch.randint(0, 2, (L[0] * L[1] * L[2],), dtype=torch.int8, device=dev, generator=g) * 2 - 1
        return {"record": np.array(_record(s.reshape(L), 0, ig.Y_GAPBC, ig.X_FREE), dtype=np.int64), "spins": s.cpu()}
    sites = case["Lx"] * case["Ly"] * case["Lz"] if case["kind"] == "film" else 0
    if case["kind"] != "film" or sites * case["sweeps"] > 1e9:
        return None  # minutes of plain array arithmetic
    return _plain_film((case["Lx"], case["Ly"], case["Lz"]), case["T"], case["H1"], case["H"], case["y"], case["x"],
                       case["init"], 0.01, seed, case["sweeps"], case["every"], dev)
