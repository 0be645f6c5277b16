"""Performance cases of the event-parallel shower library: the calls its users
make, over the range of sizes, physics settings and forms they make them in.

Kinds of case:
  run     the whole pipeline through host buffers (gaps.run): matrix element,
          shower (plain or persistent form), validation, observables,
          histograms and statistics
  jobs    an uneven multi-job batch in one persistent launch, stage by stage,
          one histogram set per job
  serve   jobs submitted to the C serving scheduler, stepped until every job's
          histograms are on the host
  shapes  the allocation-free event shapes of a caller's own events

Every output is what the call leaves for its user: the event record (momenta,
flavours, colours, links), every per-event scalar, the observables and the
histograms.  exact() computes the floating outputs with plain torch in 64
bits: Philox, the LO matrix element, the veto algorithm, the dipole map,
thrust by all planes and Durham clustering, written from their definitions.
"""
import math

import numpy as np
import torch

import paper_2403_08692_gb300 as g

DEVICE = "cuda"

# exact() covers batches up to this many events (under twenty seconds).
EXACT_EVENTS = 150_000

PHYSICS = ("sqrt_s", "t_cutoff", "alphas_mz", "n_flavours", "fixed_alphas", "trial_mode")
LEP = {"sqrt_s": 91.2, "t_cutoff": 1.0, "alphas_mz": 0.118, "n_flavours": 5, "fixed_alphas": 0, "trial_mode": 0}


def _case(kind, name=None, **kw):
    c = {"kind": kind}
    if name is not None:
        c["name"] = name
    if kind != "shapes":
        c.update(LEP)
    c.update(kw)
    return c


def _run(name, events, mode, capacity=128, layout=0, **kw):
    return _case("run", name, events=events, mode=mode, capacity=capacity, layout=layout, **kw)


PLAIN, PERSISTENT = g.SHOWER_PLAIN, g.SHOWER_PERSISTENT


def listed():
    return [
        # interactive studies and cross-checks: latency and launches count
        _run("plain_1e3", 1_000, PLAIN),
        # odd size, LEP2 energy and a low cutoff (long showers), tiled records
        _run("plain_12k_200gev", 12_347, PLAIN, layout=1, sqrt_s=200.0, t_cutoff=0.5),
        # an ordinary sample with one trial per dipole
        _run("plain_1e5_per_dipole", 100_000, PLAIN, sqrt_s=133.0, trial_mode=1),
        # the paper's headline sample: 10^6 LEP events, the default form
        _run("plain_1e6", 1_000_000, PLAIN),
        # the smallest batches a tuning loop or a test asks for
        _run("persistent_100", 100, PERSISTENT),
        # ragged size, fixed coupling, fewer flavours
        _run("persistent_20k_fixed", 20_011, PERSISTENT, n_flavours=3, fixed_alphas=1),
        # LEP2 sample, one trial per dipole, tiles of 32
        _run("persistent_3e5_200gev", 300_007, PERSISTENT, layout=2, sqrt_s=200.0, t_cutoff=2.0, trial_mode=1),
        # the headline sample in the batched form
        _run("persistent_1e6", 1_000_000, PERSISTENT),
        # a large production batch with the paper's 50 parton slots
        _run("persistent_4e6", 4_000_000, PERSISTENT, capacity=50),
        # a parameter scan: jobs of very different sizes, energies and cutoffs in one launch
        _case("jobs", "jobs_uneven_24", jobs=24, n_min=1_000, n_max=300_000, capacity=128, layout=1, mix=1),
        # the serving loop at saturation: jobs of one physics setting queued at once
        _case("serve", "serve_40", jobs=40, n_min=1_000, n_max=100_000, pool=400_000, capacity=128,
              cycles_per_round=32, mix=0),
        # event shapes of a caller's own many-particle events
        _case("shapes", "shapes_20k", events=20_000, n_lo=17, n_hi=80, capacity=96, sqrt_s=91.2),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 8 + ["jobs", "serve", "shapes"])
    if kind == "shapes":
        lo = rng.randint(2, 40)
        hi = rng.randint(lo, 100)
        return _case("shapes", events=_log_uniform(rng, 500, 40_000 if hi > 50 else 200_000), n_lo=lo, n_hi=hi,
                     capacity=hi + rng.randint(0, 28), sqrt_s=rng.choice([91.2, 133.0, 200.0]))
    physics = {"sqrt_s": rng.choice([91.2, 91.2, 133.0, 200.0]), "t_cutoff": rng.choice([0.5, 1.0, 1.0, 2.0]),
               "n_flavours": rng.choice([3, 4, 5, 5, 5]), "fixed_alphas": rng.choice([0, 0, 0, 1]),
               "trial_mode": rng.choice([0, 0, 1])}
    capacity = rng.choice([50, 64, 100, 128, 128])
    if kind == "run":
        mode = rng.choice([PLAIN, PERSISTENT])
        return _run(None, _log_uniform(rng, 100, 1_000_000), mode, capacity=capacity, layout=rng.randint(0, 2), **physics)
    if kind == "jobs":
        n_max = _log_uniform(rng, 5_000, 200_000)
        return _case("jobs", jobs=rng.randint(2, 40), n_min=rng.randint(200, 2_000), n_max=n_max, capacity=capacity,
                     layout=rng.randint(0, 2), mix=1, **physics)
    n_max = _log_uniform(rng, 5_000, 100_000)
    return _case("serve", jobs=rng.randint(4, 48), n_min=rng.randint(200, 2_000), n_max=n_max,
                 pool=n_max + rng.randint(50_000, 300_000), capacity=capacity,
                 cycles_per_round=rng.choice([8, 16, 32]), mix=rng.randint(0, 1), **physics)


# ------------------------------------------------------------------ inputs
def _physics(case):
    return {k: case[k] for k in PHYSICS}


def _jobs(case, seed):
    """The case's jobs: physics, event count and Philox seed of each.  Event
    counts are log-uniform; with mix, sqrt(s) and the cutoff differ too.  The
    mix is the case's own, the Philox keys are the seed's."""
    rng = np.random.default_rng([4, case["jobs"], case["n_min"], case["n_max"]])
    out = []
    for j in range(case["jobs"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        p = _physics(case)
        if case["mix"]:
            p["sqrt_s"] = float(rng.choice([91.2, 133.0, 200.0]))
            p["t_cutoff"] = float(rng.choice([0.5, 1.0, 2.0]))
        out.append((p, n, 1000 * seed + j))
    return out


def _synthetic_events(case, seed):
    """Massless n-parton events, n uniform in n_lo .. n_hi, by RAMBO
    (Kleiss, Stirling, Ellis, Comput. Phys. Commun. 40 (1986) 359):
    slot-major momenta and the parton counts."""
    n, cap = case["events"], case["capacity"]
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    counts = torch.randint(case["n_lo"], case["n_hi"] + 1, (n,), generator=gen, device=DEVICE, dtype=torch.int32)
    live = torch.arange(cap, device=DEVICE)[:, None] < counts[None, :]
    r = torch.rand((4, cap, n), generator=gen, device=DEVICE, dtype=torch.float64).clamp_min(1e-12)
    c = 2.0 * r[0] - 1.0
    e = torch.where(live, -torch.log(r[2] * r[3]), 0.0)
    st = torch.sqrt(1.0 - c * c)
    phi = 2.0 * math.pi * r[1]
    q = torch.stack([e * st * torch.cos(phi), e * st * torch.sin(phi), e * c])
    tot_e, tot = e.sum(0), q.sum(1)
    m = torch.sqrt(tot_e ** 2 - (tot ** 2).sum(0))
    b, x, gamma = -tot / m, case["sqrt_s"] / m, tot_e / m
    bq = (q * b[:, None]).sum(0)
    e2 = torch.where(live, x * (gamma * e + bq), 0.0)
    q2 = torch.where(live, x * (q + b[:, None] * (e + bq / (1.0 + gamma))), 0.0)
    return {"px": q2[0].contiguous(), "py": q2[1].contiguous(), "pz": q2[2].contiguous(), "e": e2.contiguous(),
            "n_partons": counts, "status": torch.full((n,), g.DONE, dtype=torch.int32, device=DEVICE)}


_TILE = {0: None, 1: 8, 2: 32}


def _record_shape(n, cap, layout, sides=1):
    T = _TILE[layout]
    if T is None:
        return (cap, n) if sides == 1 else (2, cap, n)
    tiles = (n + 31) // 32 * 32 // T
    return (tiles, cap, T) if sides == 1 else (tiles, 2, cap, T)


def _record_views(ws):
    """Views of everything a pass leaves in its workspace, in the record's own
    layout (no copies)."""
    n, cap, lay = ws.n_events, ws.capacity, ws.record_layout
    one, two = _record_shape(n, cap, lay), _record_shape(n, cap, lay, 2)
    out = {k: ws.view(k, torch.float64, one) for k in ("e", "px", "py", "pz")}
    out["flav"] = ws.view("flav", torch.int8, one)
    out["col"] = ws.view("col", torch.int16, one)
    out["acol"] = ws.view("acol", torch.int16, one)
    out["link"] = ws.view("link", torch.uint8, two)
    out.update(ws.scalars())
    out["obs"] = ws.obs()
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        ws = g.Workspace(case["events"], case["capacity"], layout=case["layout"])
        hist = torch.zeros(g.HIST_DOUBLES, dtype=torch.float64).pin_memory()
        return {"kind": kind, "mode": case["mode"], "params": g.make_params(seed=seed, **_physics(case)), "ws": ws,
                "hist": hist, "out": {"hist": hist, **_record_views(ws)}}
    if kind == "jobs":
        jobs = _jobs(case, seed)
        ws = g.Workspace(sum(n for _, n, _ in jobs), case["capacity"], layout=case["layout"])
        g.set_jobs([(g.make_params(seed=s, **p), n, 0) for p, n, s in jobs], ws)
        hist = torch.zeros((len(jobs), g.HIST_DOUBLES), dtype=torch.float64, device=DEVICE)
        return {"kind": kind, "ws": ws, "hist": hist, "out": {"hist": hist, **_record_views(ws)}}
    if kind == "serve":
        jobs = [(g.make_params(seed=s, **p), n) for p, n, s in _jobs(case, seed)]
        server = g.CServer(case["pool"], capacity=case["capacity"], max_jobs=64,
                           cycles_per_round=case["cycles_per_round"])
        return {"kind": kind, "jobs": jobs, "server": server}
    events = _synthetic_events(case, seed)
    events["obs"] = torch.empty((g.N_OBS, case["events"]), dtype=torch.float64, device=DEVICE)
    return {"kind": kind, "events": events, "n": case["events"], "capacity": case["capacity"],
            "sqrt_s": case["sqrt_s"]}


def run(state):
    kind = state["kind"]
    if kind == "run":
        rc, _ = g.run(state["params"], state["ws"], state["hist"], state["mode"])
        if rc != 0:
            raise RuntimeError(f"gaps.run: status {rc}")
        return state["out"]
    if kind == "jobs":
        ws = state["ws"]
        state["hist"].zero_()
        g.generate_me(None, ws)
        g.shower_persistent(None, ws)
        g.validate(None, ws)
        g.observables(None, ws)
        g.histograms(None, ws, state["hist"])
        return state["out"]
    if kind == "serve":
        server = state["server"]
        index = {server.submit(p, n): k for k, (p, n) in enumerate(state["jobs"])}
        hists = np.zeros((len(index), g.HIST_DOUBLES))
        left = len(index)
        while left:
            for jid in server.step():
                hists[index[jid]] = server.poll(jid)
                left -= 1
        return hists
    ev = state["events"]
    g.event_shapes_noalloc(ev["px"], ev["py"], ev["pz"], ev["e"], ev["n_partons"], ev["status"], state["n"],
                           state["capacity"], state["sqrt_s"], ev["obs"])
    return ev["obs"]


# -------------------------------------------------------------------- work
def _per_event(case, sqrt_s, t_cutoff):
    """(bytes, flops) an event cannot do without: the finished record (44
    bytes a parton), the per-event scalars and observables (150 bytes); in FP64
    flops, 40 per winning trial (logarithm and update) and 940 per emission
    (kinematics and the dipoles it moves).  Winners and emissions per event
    grow about as the square of L = ln(s / 4 t_C): 30 and 2.9 at L = 7.6 (LEP,
    t_C = 1 GeV^2)."""
    grow = (math.log(sqrt_s ** 2 / (4.0 * t_cutoff)) / 7.64) ** 2
    winners, emissions = 30.0 * grow, 2.9 * grow
    return 44.0 * (2.0 + emissions) + 150.0, 40.0 * winners + 940.0 * emissions


def work(case):
    if case["kind"] == "run":
        b, f = _per_event(case, case["sqrt_s"], case["t_cutoff"])
        return {"bytes": b * case["events"] + 8 * g.HIST_DOUBLES, "flops": f * case["events"]}
    if case["kind"] in ("jobs", "serve"):
        total = {"bytes": 0.0, "flops": 0.0}
        for p, n, _ in _jobs(case, 1):
            b, f = _per_event(case, p["sqrt_s"], p["t_cutoff"])
            total["bytes"] += b * n + 8 * g.HIST_DOUBLES
            total["flops"] += f * n
        return total
    # shapes: momenta in, observables out; the thrust axis needs every pair's
    # plane once (about 20 operations a pair), the clustering every pair's
    # distance once and the merged jet's at each merge (about 10 each)
    n = (case["n_lo"] + case["n_hi"]) / 2.0
    return {"bytes": case["events"] * (32.0 * n + 8 + 8 * g.N_OBS), "flops": case["events"] * 20.0 * n * n}


def tolerance(case):
    # FP64 throughout.  Against exact() the records differ by up to 3.5e-13 (2-norm;
    # ten emissions amplify the rounding, most at 200 GeV), the event shapes by
    # 4e-15 with square roots good to 1.5e-13.  Decisions agree event by event
    # but for trials that tie within the rounding; histograms are exact sums.
    if case["kind"] == "shapes":
        return {"rel": 1e-13, "max": 1e-11}
    if case["kind"] == "serve":
        return {"rel": 1e-12, "max": 1e-11}
    return {"rel": 2e-12, "max": 1e-9, "differ": 1e-5}


# ------------------------------------------------------------------- exact
# The definitions in plain torch, 64 bits.
PI = math.pi
CF, CA, TR, NC = 4.0 / 3.0, 3.0, 0.5, 3.0
M_Z, GAMMA_Z, ALPHA_QED, SIN2W, GEV2_TO_PB = 91.1876, 2.4952, 1.0 / 128.802, 0.222, 0.389379e9
DRAW_ME, DRAW_TRIAL, DRAW_WINNER = 1, 2, 3
MASK32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) on int64 tensors."""
    k0, k1 = seed & MASK32, (seed >> 32) & MASK32
    like = c0 + c1 + c2 + c3
    c0, c1, c2, c3 = (torch.zeros_like(like) + c for c in (c0, c1, c2, c3))
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & MASK32) ^ c1 ^ k0, p1 & MASK32, ((p0 >> 32) & MASK32) ^ c3 ^ k1, p0 & MASK32)
        k0, k1 = (k0 + 0x9E3779B9) & MASK32, (k1 + 0xBB67AE85) & MASK32
    return c0, c1, c2, c3


def _uniforms(ids, step, slot, purpose, seed):
    """The two 52-bit uniforms of one Philox block."""
    w = _philox(ids, torch.full_like(ids, step) if isinstance(step, int) else step, slot, torch.full_like(ids, purpose),
                seed)
    unit = lambda hi, lo: (2.0 * (((hi >> 6) << 26) | (lo >> 6)).double() + 1.0) * 2.0 ** -53
    return unit(w[0], w[1]), unit(w[2], w[3])


def _choose(mask, a, b):
    """a where mask, else b, in 64 bits."""
    two = torch.tensor([b, a], dtype=torch.float64, device=mask.device)
    return two[mask.long()]


def _alpha_s(p, t):
    if p["fixed_alphas"]:
        return torch.full_like(t, p["alphas_mz"])
    b0 = (33.0 - 2.0 * p["n_flavours"]) / (12.0 * PI)
    return p["alphas_mz"] / (1.0 + p["alphas_mz"] * b0 * torch.log(t / M_Z ** 2))


def _mdot(a, b):
    return a[..., 0] * b[..., 0] - a[..., 1] * b[..., 1] - a[..., 2] * b[..., 2] - a[..., 3] * b[..., 3]


def _matrix_element(p, seed, ids):
    """App. B: flavour, direction and weight of every event."""
    zero = torch.zeros_like(ids)
    u0, u1 = _uniforms(ids, 0, zero, DRAW_ME, seed)
    v0, _ = _uniforms(ids, 0, zero + 1, DRAW_ME, seed)
    nf, s = p["n_flavours"], p["sqrt_s"] ** 2
    flav = (1 + (u0 * nf).long()).clamp_max(nf)
    cth = 2.0 * u1 - 1.0
    sth, phi, e = torch.sqrt(1.0 - cth * cth), 2.0 * PI * v0, 0.5 * p["sqrt_s"]
    quark = torch.stack([torch.full_like(cth, e), e * sth * torch.cos(phi), e * sth * torch.sin(phi), e * cth], -1)
    anti = torch.cat([quark[:, :1], -quark[:, 1:]], -1)
    up = (flav == 2) | (flav == 4)
    q = _choose(up, 2.0 / 3.0, -1.0 / 3.0)
    a = _choose(up, 0.5, -0.5)
    v = a - 2.0 * q * SIN2W
    ae, ve = -0.5, -0.5 + 2.0 * SIN2W
    kappa = 1.0 / (4.0 * SIN2W * (1.0 - SIN2W))
    den = (s - M_Z ** 2) ** 2 + (GAMMA_Z * M_Z) ** 2
    chi1, chi2 = kappa * s * (s - M_Z ** 2) / den, kappa ** 2 * s * s / den
    even = q * q - 2.0 * q * ve * v * chi1 + (ae ** 2 + ve ** 2) * (a * a + v * v) * chi2
    odd = -2.0 * q * ae * a * chi1 + 4.0 * ae * ve * a * v * chi2
    pref = PI * ALPHA_QED ** 2 / (2.0 * s) * NC * GEV2_TO_PB
    weight = nf * 2.0 * pref * ((1.0 + cth * cth) * even + 2.0 * cth * odd)
    return flav, quark, anti, weight


def _det3(a, b, c):
    return (a[0] * (b[1] * c[2] - b[2] * c[1]) - a[1] * (b[0] * c[2] - b[2] * c[0])
            + a[2] * (b[0] * c[1] - b[1] * c[0]))


def _complement(a, b, c):
    """N with N.X = det[X; a; b; c]."""
    A, B, C = a.unbind(-1), b.unbind(-1), c.unbind(-1)
    pick = lambda r: ([A[i] for i in r], [B[i] for i in r], [C[i] for i in r])
    return torch.stack([_det3(*pick((1, 2, 3))), _det3(*pick((0, 2, 3))), -_det3(*pick((0, 1, 3))),
                        _det3(*pick((0, 1, 2)))], -1)


def _dipole_map(a, b, z, y, phi):
    """Catani-Seymour final-final map of massless splitter a, spectator b."""
    ab = _mdot(a, b)
    n1 = None
    for r in (1, 2, 3):
        ref = torch.zeros_like(a)
        ref[:, 0] = 1.0
        ref[:, r] = 1.0
        n = ref - (_mdot(ref, b) / ab)[:, None] * a - (_mdot(ref, a) / ab)[:, None] * b
        if n1 is None:
            n1, open_ = n, _mdot(n, n).abs() < 1e-4
        else:
            n1 = torch.where(open_[:, None], n, n1)
            open_ = open_ & (_mdot(n, n).abs() < 1e-4)
    n1 = n1 / torch.sqrt(-_mdot(n1, n1))[:, None]
    n2 = _complement(a, b, n1)
    n2 = n2 / torch.sqrt(-_mdot(n2, n2))[:, None]
    kt = torch.sqrt(z * (1.0 - z) * y * 2.0 * ab)
    k = (kt * torch.cos(phi))[:, None] * n1 + (kt * torch.sin(phi))[:, None] * n2
    z, y = z[:, None], y[:, None]
    return z * a + (1.0 - z) * y * b + k, (1.0 - z) * a + z * y * b - k, (1.0 - y) * b


def _shower(p, seed, ids, cap):
    """The serial veto algorithm (Sec. 2, App. A, App. C), every event of the
    batch in step.  Returns momenta [n][cap][4] (zero beyond the partons),
    parton counts, finished flags, final scales and weights."""
    n_ev, nf, tc = ids.numel(), p["n_flavours"], p["t_cutoff"]
    per_dipole = p["trial_mode"] == 1
    K = nf + 1
    dev = ids.device
    as2pi = float(_alpha_s(p, torch.tensor([tc], dtype=torch.float64))) / (2.0 * PI)
    me_flav, quark, anti, weight = _matrix_element(p, seed, ids)
    mom = torch.zeros((n_ev, cap, 4), dtype=torch.float64, device=dev)
    mom[:, 0], mom[:, 1] = quark, anti
    gluon = torch.zeros((n_ev, cap), dtype=torch.bool, device=dev)
    link = torch.full((n_ev, cap, 2), -1, dtype=torch.long, device=dev)
    link[:, 0, 0], link[:, 1, 1] = 1, 0
    n = torch.full((n_ev,), 2, dtype=torch.long, device=dev)
    lnt = torch.full((n_ev,), math.log(p["sqrt_s"] ** 2), dtype=torch.float64, device=dev)
    t_end = torch.full((n_ev,), tc, dtype=torch.float64, device=dev)
    done = torch.ones(n_ev, dtype=torch.bool, device=dev)
    act = torch.arange(n_ev, device=dev)
    step = 0
    while act.numel():
        A, M = act.numel(), int(n[act].max())
        P, lk, gl, idA = mom[act, :M], link[act, :M], gluon[act, :M], ids[act]
        partner = torch.gather(P[:, :, None, :].expand(A, M, 2, 4), 1, lk.clamp_min(0)[..., None].expand(A, M, 2, 4))
        q2 = 2.0 * _mdot(P[:, :, None, :], partner)
        ok = (lk >= 0) & (q2 >= 4.0 * tc)
        zp = 0.5 * (1.0 + torch.sqrt((1.0 - 4.0 * tc / torch.where(ok, q2, 8.0 * tc))))
        zm = 1.0 - zp
        ls = torch.log(zp / zm)
        g2 = gl[:, :, None].expand(A, M, 2)
        c_qq = as2pi * 0.5 * TR * (zp - zm)
        c0 = as2pi * ls * _choose(g2, CA, 2.0 * CF)
        d = 2 * torch.arange(M, device=dev)[:, None] + torch.arange(2, device=dev)
        if per_dipole:
            c_sum = torch.where(g2, c0 + nf * c_qq, c0)
            u, _ = _uniforms(idA[:, None, None].expand(A, M, 2).contiguous(), step,
                             (4 * d)[None].expand(A, M, 2).contiguous(), DRAW_TRIAL, seed)
            lt = torch.where(ok, lnt[act][:, None, None] + torch.log(u) / c_sum, -math.inf)
            best, arg = lt.reshape(A, -1).max(1)
            kap = torch.zeros_like(arg)
        else:
            blocks = (K + 1) // 2
            slot = (4 * d)[:, :, None] + torch.arange(blocks, device=dev)
            u = torch.stack(_uniforms(idA[:, None, None, None].expand(A, M, 2, blocks).contiguous(), step,
                                      slot[None].expand(A, M, 2, blocks).contiguous(), DRAW_TRIAL, seed), -1)
            u = u.reshape(A, M, 2, 2 * blocks)[..., :K]
            c = torch.where(torch.arange(K, device=dev) == 0, c0[..., None], c_qq[..., None])
            allowed = ok[..., None] & (g2[..., None] | (torch.arange(K, device=dev) == 0))
            lt = torch.where(allowed, lnt[act][:, None, None, None] + torch.log(u) / c, -math.inf)
            best, arg = lt.reshape(A, -1).max(1)
            kap, arg = arg % K, arg // K
        won = best > math.log(tc)
        done_now = act[~won]
        act, best, arg, kap, row = act[won], best[won], arg[won], kap[won], torch.nonzero(won)[:, 0]
        del done_now
        if act.numel() == 0:
            break
        lnt[act] = best
        i, side = arg // 2, arg % 2
        at = lambda x: x[row, i, side]
        wq2, wzp, wls, wk, wg = at(q2), at(zp), at(ls), at(lk), at(g2)
        wzm = 1.0 - wzp
        idW = ids[act]
        zero = torch.zeros_like(idW)
        rz, rv = _uniforms(idW, step, zero, DRAW_WINNER, seed)
        rphi, rk = _uniforms(idW, step, zero + 1, DRAW_WINNER, seed)
        if per_dipole:
            cq, cg = at(c_qq), at(c0)
            target = rk * (cg + nf * cq)
            kap = torch.where(wg & (target >= cg), 1 + ((target - cg) / cq).long().clamp(0, nf - 1), 0)
        soft = kap == 0
        one_z = torch.where(soft, wzp * torch.exp(-rz * wls), wzp - (wzp - wzm) * rz)
        z = torch.where(soft, wzm - wzp * torch.expm1(-rz * wls), wzm + (wzp - wzm) * rz)
        t = torch.exp(best)
        y = t / (wq2 * z * one_z)
        den = one_z + z * y
        val = torch.where(~wg, CF * (2.0 / den - (1.0 + z)),
                          torch.where(soft, 0.5 * CA * (2.0 / den - 2.0 + z * one_z),
                                      0.5 * TR * (1.0 - 2.0 * z * one_z)))
        over = torch.where(~wg, 2.0 * CF / one_z, torch.where(soft, CA / one_z, 0.5 * TR))
        acc = (y < 1.0) & (rv < (1.0 - y) * _alpha_s(p, t) * val / (2.0 * PI * as2pi * over))
        full = acc & (n[act] >= cap)
        t_end[act[full]] = t[full]
        done[act[full]] = False
        emit = acc & ~full
        if bool(emit.any()):
            ev, si, sk, ss, kp = act[emit], i[emit], wk[emit], side[emit], kap[emit]
            pi, pj, pk = _dipole_map(mom[ev, si], mom[ev, sk], z[emit], y[emit], 2.0 * PI * rphi[emit])
            j = n[ev]
            mom[ev, si], mom[ev, j], mom[ev, sk] = pi, pj, pk
            split = kp > 0  # g -> q qbar: the antiquark takes the anticolour line
            e, a, b = ev[split], si[split], j[split]
            q = link[e, a, 1]
            gluon[e, a] = False
            link[e, a, 1], link[e, b, 0], link[e, b, 1], link[e, q, 0] = -1, -1, q, b
            e, a, b, k, sd = ev[~split], si[~split], j[~split], sk[~split], ss[~split]
            gluon[e, b] = True  # the gluon goes between splitter and spectator
            link[e, a, sd], link[e, b, sd], link[e, b, 1 - sd], link[e, k, 1 - sd] = b, k, a, b
            n[ev] += 1
        act = act[~full]
        step += 1
    return mom, n, done, t_end, weight


def _event_shapes(mom, n, sqrt_s):
    """Observables [n_events][8] of momenta [n_events][slots][4] (E, p): y23,
    y34, y45, y56, 1 - T, rho_H, B_T, B_W."""
    s = sqrt_s ** 2
    out = torch.full((mom.shape[0], 8), -1.0, dtype=torch.float64, device=mom.device)
    for m in torch.unique(n).tolist():
        rows = torch.nonzero(n == m)[:, 0]
        pairs = torch.combinations(torch.arange(m, device=mom.device)) if m > 2 else None
        chunk = max(1, int(2e7 / max(1, m * m * m // 2)))
        for r in rows.split(chunk):
            out[r] = _shapes_of(mom[r, :m], m, pairs, s)
    return out


def _shapes_of(p, m, pairs, s):
    N, v = p.shape[0], p[..., 1:]
    mag = v.norm(dim=-1)
    axis = v[:, 0]
    if m > 2:
        j, k = pairs[:, 0], pairs[:, 1]
        normal = torch.linalg.cross(v[:, j], v[:, k])
        sign = _choose(normal @ v.transpose(1, 2) >= 0.0, 1.0, -1.0)
        at = torch.arange(j.numel(), device=p.device)
        sign[:, at, j] = 0.0
        sign[:, at, k] = 0.0
        rest = sign @ v
        best = torch.full((N,), -1.0, dtype=torch.float64, device=p.device)
        flat = (normal == 0.0).all(-1)
        for a in (1.0, -1.0):
            for b in (1.0, -1.0):
                c = rest + a * v[:, j] + b * v[:, k]
                score, where = torch.where(flat, -1.0, (c * c).sum(-1)).max(1)
                axis = torch.where((score > best)[:, None], c[torch.arange(N, device=p.device), where], axis)
                best = torch.maximum(best, score)
        thrust = torch.where(best >= 0.0, torch.sqrt(best.clamp_min(0.0)) / mag.sum(1), 1.0)
    else:
        thrust = torch.ones(N, dtype=torch.float64, device=p.device)
    axis = axis / axis.norm(dim=-1, keepdim=True)
    plus = ((v * axis[:, None]).sum(-1) >= 0.0)[..., None]
    mass = lambda h: h[:, 0] ** 2 - (h[:, 1:] ** 2).sum(-1)
    heavy = torch.maximum(mass((p * plus).sum(1)), mass((p * ~plus).sum(1)))
    pt = torch.linalg.cross(v, axis[:, None].expand_as(v)).norm(dim=-1)
    bp = (pt * plus[..., 0]).sum(1) / (2.0 * mag.sum(1))
    bm = (pt * ~plus[..., 0]).sum(1) / (2.0 * mag.sum(1))
    y = torch.full((N, 4), -1.0, dtype=torch.float64, device=p.device)
    jets, row = p.clone(), torch.arange(N, device=p.device)
    for q in range(m, 2, -1):
        e, w = jets[:, :q, 0], jets[:, :q, 1:]
        unit = w / w.norm(dim=-1, keepdim=True)
        # 1 - cos = |u_i - u_j|^2 / 2, free of cancellation
        dist = 0.5 * ((unit[:, :, None] - unit[:, None]) ** 2).sum(-1)
        yy = 2.0 * torch.minimum(e[:, :, None], e[:, None]) ** 2 * dist / s
        yy = torch.where(torch.ones(q, q, device=p.device).triu(1).bool(), yy, math.inf).reshape(N, -1)
        least, arg = yy.min(1)
        if q <= 6:
            y[:, q - 3] = least
        a, b = arg // q, arg % q
        jets[row, a] = jets[row, a] + jets[row, b]
        jets[row, b] = jets[:, q - 1].clone()
    return torch.cat([y, torch.stack([1.0 - thrust, heavy / s, bp + bm, torch.maximum(bp, bm)], -1)], -1)


def _histograms(obs, weight, done):
    """Sum w, sum w^2 and entries of every cell, [8][102][3]."""
    hist = torch.zeros((8, 102, 3), dtype=torch.float64, device=obs.device)
    for h in range(8):
        o = obs[:, h]
        if h < 4:
            use, x, lo, hi = done & (o > 0.0), torch.log10(o.clamp_min(1e-300)), -4.3, -0.3
        else:
            use, x, lo, hi = done, o.clamp_min(0.0), 0.0, 0.5 if h < 6 else 0.4
        f = (x - lo) / (hi - lo) * 100
        cell = torch.where(f < 0.0, 0, torch.where(f >= 100, 101, 1 + f.clamp(0, 99).long()))[use]
        w = weight[use]
        for k, val in enumerate((w, w * w, torch.ones_like(w))):
            hist[h, :, k] = torch.zeros(102, dtype=torch.float64, device=obs.device).index_add_(0, cell, val)
    return hist.reshape(-1)


def _pass(p, seed, n, cap):
    """One job's events, observables and histograms."""
    got = []
    for ids in torch.arange(n, device=DEVICE).split(25_000):
        mom, k, done, t, weight = _shower(p, seed, ids, cap)
        obs = torch.where(done[:, None], _event_shapes(mom, k, p["sqrt_s"]), -1.0)
        got.append((mom, done, t, weight, obs))
    mom, done, t, weight, obs = (torch.cat(x) for x in zip(*got))
    return {"mom": mom, "t": t, "weight": weight, "obs": obs, "hist": _histograms(obs, weight, done)}


def _in_layout(x, layout, cap):
    """[n][cap] values in the record layout (zero in the padding)."""
    T = _TILE[layout]
    if T is None:
        return x.T.contiguous()
    n = x.shape[0]
    pad = torch.zeros(((n + 31) // 32 * 32, cap), dtype=x.dtype, device=x.device)
    pad[:n] = x
    return pad.reshape(-1, T, cap).transpose(1, 2).contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "shapes":
        ev = _synthetic_events(case, seed)
        mom = torch.stack([ev[c] for c in ("e", "px", "py", "pz")], -1).transpose(0, 1)
        return _event_shapes(mom, ev["n_partons"].long(), case["sqrt_s"]).T.contiguous()
    jobs = _jobs(case, seed) if kind != "run" else [(_physics(case), case["events"], seed)]
    if sum(n for _, n, _ in jobs) > EXACT_EVENTS:
        return None
    if kind == "serve":
        return np.stack([_pass(p, s, n, case["capacity"])["hist"].cpu().numpy() for p, n, s in jobs])
    done = [_pass(p, s, n, case["capacity"]) for p, n, s in jobs]
    whole = {k: torch.cat([d[k] for d in done]) for k in ("mom", "t", "weight", "obs")}
    out = {k: _in_layout(whole["mom"][..., c], case["layout"], case["capacity"])
           for c, k in enumerate(("e", "px", "py", "pz"))}
    out.update(t=whole["t"], weight=whole["weight"], obs=whole["obs"].T.contiguous())
    out["hist"] = torch.stack([d["hist"] for d in done]) if kind == "jobs" else done[0]["hist"]
    return out
