"""The work that a user of this library has it do, as cases that can be timed and compared.

Five ways in, each through the package's public entry points, over the sizes
that the configurations, the tests and the benchmark of this repository use:

  lattice  one lattice on its own context: sweeps of a schedule, then E/N and
           the spins (a measurement loop; the chain goes on from pass to pass)
  custom   a schedule built by hand from single half-sweeps, a renormalisation
           and the energy of caller-held arrays
  solve    a whole solve: a new lattice, couplings uploaded from pinned host
           memory, sweeps, E/N and spins back on the host
  pool     many independent lattices swept together, then every E/N and all
           spins
  serve    the continuous-batching request loop over a fixed list of requests

``exact`` computes the same chains in 64 bits with plain torch.
"""
import math

import torch

from paper_1006_2566_gb300 import hsg, serve

_UPDATES = {"none": hsg.HSG_NONE, "met": hsg.HSG_METROPOLIS, "hb": hsg.HSG_HEATBATH, "met_or": hsg.HSG_METROPOLIS_OR}
_PROPOSALS = {"sphere": hsg.HSG_PROP_SPHERE, "ball": hsg.HSG_PROP_BALL}
# Threads, sites per tile, CTAs per SM and hits per pass of a served pool: a
# server tunes once at start-up and passes the result on.
_SERVE_CONFIG = (256, 1024, 16, 0)

_streams = {}


def _stream():
    """The one CUDA stream that this program runs the library on."""
    d = torch.cuda.current_device()
    if d not in _streams:
        _streams[d] = torch.cuda.Stream()
    return _streams[d]


def listed():
    return [
        # The smallest: a lone L = 16 sample, 1-hit Metropolis with a uniform-sphere proposal at T = 1, ten sweeps
        # and a measurement.  Latency and launches are all there is.
        _lattice("lone L=16 Metropolis", 16, "met", "sphere", hits=1, n_or=0, T=1.0, sweeps=10, cadence=0),
        # A small lattice by heat-bath and over-relaxation, as in equilibration runs of one sample.
        _lattice("lone L=40 heat-bath + 2 OR", 40, "hb", "sphere", hits=1, n_or=2, T=0.6, sweeps=10, cadence=5),
        # An odd half-row (33 sites of a colour): the fused Metropolis + reflection pass.
        _lattice("lone L=66 fused pass", 66, "met_or", "ball", hits=4, n_or=0, T=0.5, sweeps=5, cadence=5),
        # The paper's size: 4-hit Metropolis and one over-relaxation sweep, the state in L2.
        _lattice("lone L=128 Metropolis + OR", 128, "met", "ball", hits=4, n_or=1, T=0.5, sweeps=10, cadence=10),
        # The benchmark's lattice: heat-bath and four over-relaxation sweeps, streaming from HBM.
        _lattice("lone L=256 heat-bath + 4 OR", 256, "hb", "sphere", hits=1, n_or=4, T=0.3, sweeps=10, cadence=10),
        # The 12-byte spin layout, at a ragged size.
        _lattice("packed L=130 heat-bath + 2 OR", 130, "hb", "sphere", hits=1, n_or=2, T=0.8, sweeps=2, cadence=2,
                 layout="packed"),
        # A schedule of the user's own from single half-sweeps, energy of caller-held arrays.
        {"name": "half-sweeps L=100", "way": "custom", "L": 100, "update": "met", "proposal": "ball", "hits": 2,
         "n_or": 1, "T": 0.7, "sweeps": 3, "cadence": 1, "layout": "float4"},
        # A first and only pass on a new sample: couplings in fp64 from the host, results back to the host.
        {"name": "solve L=48", "way": "solve", "L": 48, "update": "met", "proposal": "ball", "hits": 4, "n_or": 2,
         "T": 0.6, "sweeps": 50, "cadence": 10, "layout": "float4", "j64": True},
        # The same at a size where the copies and the layout conversion weigh: one lattice streamed in and out.
        {"name": "solve L=192", "way": "solve", "L": 192, "update": "hb", "proposal": "sphere", "hits": 1, "n_or": 4,
         "T": 0.3, "sweeps": 1, "cadence": 1, "layout": "float4", "j64": False},
        # Many samples and replicas of uneven L with a temperature ramp, autotuned.
        _pool("pool of 256, L=16..48", 128, 2, "16,24,32,48", "met", "ball", hits=4, n_or=2, sweeps=10, cadence=10,
              tune=True),
        # Many samples of one small lattice.
        _pool("pool of 128, L=16", 128, 1, "16", "met", "sphere", hits=1, n_or=0, sweeps=50, cadence=0, tune=False),
        # The request loop, all requests waiting: sides, temperatures and sweep counts spread as in the serving
        # workload.
        {"name": "serve 48 requests", "way": "serve", "requests": 48, "sides": "16,24,32,40,48,56,64,72,80,88,96",
         "update": "met", "proposal": "ball", "hits": 4, "n_or": 2, "cadence": 10, "lo": 50, "hi": 500},
    ]


def _lattice(name, L, update, proposal, hits, n_or, T, sweeps, cadence, layout="float4"):
    return {"name": name, "way": "lattice", "L": L, "update": update, "proposal": proposal, "hits": hits, "n_or": n_or,
            "T": T, "sweeps": sweeps, "cadence": cadence, "layout": layout}


def _pool(name, samples, replicas, sides, update, proposal, hits, n_or, sweeps, cadence, tune):
    return {"name": name, "way": "pool", "samples": samples, "replicas": replicas, "sides": sides, "update": update,
            "proposal": proposal, "hits": hits, "n_or": n_or, "sweeps": sweeps, "cadence": cadence, "tune": tune}


def _log_even(rng, lo, hi):
    """An even number between lo and hi, spread over the logarithm."""
    return 2 * max(lo // 2, min(hi // 2, int(round(math.exp(rng.uniform(math.log(lo / 2), math.log(hi / 2)))))))


def draw(rng):
    way = rng.choice(["lattice", "lattice", "lattice", "lattice", "custom", "solve", "pool", "pool", "serve"])
    update = rng.choice(["met", "met", "hb", "hb", "met_or", "none"])
    hits = rng.randint(1, 5) if update in ("met", "met_or") else 1
    c = {"way": way, "update": update, "proposal": rng.choice(["sphere", "ball"]), "hits": hits,
         "n_or": rng.randint(1 if update == "none" else 0, 4), "cadence": rng.choice([0, 1, 3, 10])}
    if way in ("lattice", "custom", "solve"):
        L = _log_even(rng, 4, 256 if way == "lattice" else 200)
        c.update(L=L, T=round(rng.uniform(0.2, 1.0), 3), sweeps=rng.randint(1, 10),
                 layout=rng.choice(["float4", "float4", "float4", "packed"]))
        if way == "custom" and update == "none":
            c.update(update="hb")
        if way == "solve":
            c.update(j64=rng.random() < 0.3, sweeps=rng.randint(5, 50) if L <= 100 else rng.randint(1, 5))
        return c
    if way == "pool":
        sides = sorted({_log_even(rng, 4, 96) for _ in range(rng.randint(1, 4))})
        mean = sum(L ** 3 for L in sides) / len(sides)
        n = max(8, min(256, int(9e6 / mean * rng.uniform(0.3, 1.0))))
        c.update(samples=max(4, n // 2), replicas=rng.choice([1, 2]), sides=",".join(map(str, sides)),
                 sweeps=rng.randint(3, 20), tune=rng.random() < 0.5)
        return c
    lo = rng.randint(10, 100)
    c.update(requests=rng.randint(8, 24), sides=",".join(map(str, sorted({_log_even(rng, 8, 96) for _ in range(6)}))),
             lo=lo, hi=lo + rng.randint(20, 350))
    return c


def _sides(case):
    return [int(x) for x in case["sides"].split(",")]


def _specs(case, seed):
    """(L, seed, sample, replica, T) of every lattice of a pool: the samples
    take the sides in turn and ramp T from 0.2 to 1."""
    sides, n = _sides(case), case["samples"]
    return [(sides[s % len(sides)], seed, s, r, 0.2 + 0.8 * s / max(1, n - 1))
            for s in range(n) for r in range(case["replicas"])]


def _requests(case, seed):
    """The requests of a served case: sides in turn, sweep counts and
    temperatures spread evenly over their ranges, all waiting at the start."""
    sides, n = _sides(case), case["requests"]
    return [serve.Request(k, 0.0, sides[k % len(sides)], seed, k, 0.2 + 0.8 * ((7 * k) % n) / n,
                          case["lo"] + (case["hi"] - case["lo"]) * ((5 * k) % n) // n) for k in range(n)]


def _schedule_kw(case):
    return dict(kind=_UPDATES[case["update"]], hits=case["hits"], proposal=_PROPOSALS[case["proposal"]], step=0.5,
                n_or=case["n_or"], renorm_every=case["cadence"])


def _couplings(case, seed):
    """Gaussian couplings on the device, site-major, fp32 values."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 31) + case["L"])
    return torch.randn(3 * case["L"] ** 3, generator=g, device="cuda", dtype=torch.float32)


def _layout(case):
    return hsg.HSG_LAYOUT_PACKED if case["layout"] == "packed" else hsg.HSG_LAYOUT_FLOAT4


def prepare(case, seed):
    way, stream = case["way"], _stream()
    st = {"case": case, "stream": stream}
    if way in ("lattice", "custom"):
        L = case["L"]
        J = _couplings(case, seed)
        st["J"] = J
        st["spins"] = torch.empty(3 * L ** 3, device="cuda", dtype=torch.float32)
        st["e"] = torch.empty(1, device="cuda", dtype=torch.float64)
        stream.wait_stream(torch.cuda.current_stream())
        lat = hsg.Lattice(L, int(seed), 1, 0, stream, _layout(case))
        lat.set_couplings(J)
        st["lat"] = lat
        st["sched"] = hsg.schedule(T=case["T"], **_schedule_kw(case))
    elif way == "solve":
        J = _couplings(case, seed)
        J = J.double() if case["j64"] else J
        st["J"] = torch.empty(J.shape, dtype=J.dtype, pin_memory=True).copy_(J)
        st["spins"] = torch.empty(J.numel(), dtype=torch.float32, pin_memory=True)
        st["seed"] = int(seed)
        st["sched"] = hsg.schedule(T=case["T"], **_schedule_kw(case))
    elif way == "pool":
        specs = _specs(case, int(seed))
        budget = sum((28 * L ** 3 + 255) // 256 * 256 for L, *_ in specs)
        pool = hsg.Pool(budget, len(specs), stream)
        st["slots"] = [pool.admit(*spec) for spec in specs]
        st["spins"] = torch.empty(sum(3 * L ** 3 for L, *_ in specs), device="cuda", dtype=torch.float32)
        st["parts"] = list(st["spins"].split([3 * L ** 3 for L, *_ in specs]))
        st["pool"], st["sched"] = pool, hsg.schedule(**_schedule_kw(case))
        if case["tune"]:
            hsg.hsg_pool_autotune(pool.pool, st["sched"])
    else:
        st["requests"] = _requests(case, int(seed))
        st["budget"] = sum((28 * r.L ** 3 + 255) // 256 * 256 for r in st["requests"])
    return st


def run(st):
    case, way = st["case"], st["case"]["way"]
    if way == "lattice":
        lat = st["lat"]
        lat.sweep(st["sched"], case["sweeps"])
        e = lat.energy()
        hsg.hsg_get_spins(lat.ctx, st["spins"])
        return {"energy": e, "spins": st["spins"]}
    if way == "custom":
        lat, sched = st["lat"], st["sched"]
        for _ in range(case["sweeps"]):
            for colour in (0, 1):
                lat.half_sweep(sched, _UPDATES[case["update"]], colour)
            for _ in range(case["n_or"]):
                for colour in (0, 1):
                    lat.half_sweep(sched, hsg.HSG_OVERRELAX, colour)
            k = lat.sweep_count + 1
            lat.sweep_count = k
            if case["cadence"] and k % case["cadence"] == 0:
                lat.renorm()
        hsg.hsg_get_spins(lat.ctx, st["spins"])
        hsg.hsg_energy_noalloc(case["L"], st["spins"], st["J"], st["e"], st["stream"])
        return {"energy": st["e"], "spins": st["spins"]}
    if way == "solve":
        with hsg.Lattice(case["L"], st["seed"], 1, 0, st["stream"], _layout(case)) as lat:
            lat.set_couplings(st["J"])
            lat.sweep(st["sched"], case["sweeps"])
            e = lat.energy()
            hsg.hsg_get_spins(lat.ctx, st["spins"])
        return {"energy": e, "spins": st["spins"]}
    if way == "pool":
        pool = st["pool"]
        pool.sweep(st["sched"], case["sweeps"])
        e = pool.energies()
        for slot, part in zip(st["slots"], st["parts"]):
            hsg.hsg_pool_get_spins(pool.pool, slot, part)
        return {"energies": e, "spins": st["spins"]}
    results, _ = serve.serve(st["requests"], _schedule_kw(case), st["budget"], len(st["requests"]), st["stream"],
                             config=_SERVE_CONFIG)
    return {"energies": torch.tensor([r.energy for r in sorted(results, key=lambda r: r.rid)], dtype=torch.float64)}


# Floating-point operations of one site update (a product, sum, division or
# elementary function each count one): field 33, reflection 16, a Metropolis
# hit about 45, a heat-bath draw about 60.
_FIELD, _REFLECT, _HIT, _BATH = 33, 16, 45, 60


def _flops_per_sweep(case):
    main = {"none": 0, "met": _FIELD + _HIT * case["hits"], "hb": _FIELD + _BATH,
            "met_or": _FIELD + _HIT * case["hits"] + _REFLECT}[case["update"]]
    return main + case["n_or"] * (_FIELD + _REFLECT)


def work(case):
    way = case["way"]
    if way in ("lattice", "custom"):  # spins and couplings in, spins out
        n = case["L"] ** 3
        return {"bytes": 36 * n, "flops": n * (case["sweeps"] * _flops_per_sweep(case) + 25)}
    if way == "solve":  # couplings in, spins out
        n = case["L"] ** 3
        return {"bytes": n * (12 + (24 if case["j64"] else 12)), "flops": n * (case["sweeps"] * _flops_per_sweep(case) + 25)}
    if way == "pool":
        n = sum(L ** 3 for L, *_ in _specs(case, 0))
        return {"bytes": 36 * n, "flops": n * (case["sweeps"] * _flops_per_sweep(case) + 25)}
    # the state of every request is made, swept and measured on the device
    reqs = _requests(case, 0)
    return {"bytes": 24 * sum(r.L ** 3 for r in reqs),
            "flops": sum(r.L ** 3 * (r.sweeps * _flops_per_sweep(case) + 25) for r in reqs)}


def _growth(case):
    """How many times a difference between two chains grows, in passes that
    each multiply it by about 4 (measured: a reflection sweep 3.8 times, a
    Metropolis or heat-bath sweep about 2)."""
    per_sweep = case["n_or"] + (case["update"] == "met_or") + 0.5 * (case["update"] in ("met", "hb"))
    return case["sweeps"] * per_sweep


def _comparable(case):
    """Whether two fp32 chains of this case stay close.  The dynamics are
    chaotic: rounding differences of 1e-7 grow by about 4 with each
    reflection sweep until one Metropolis decision or one heat-bath frame
    falls the other way, and soon after that the chains share their
    distribution only."""
    if case["way"] == "serve":
        return False
    return _growth(case) <= 5.5 or (case["update"] == "met" and case["n_or"] == 0 and case["sweeps"] <= 50)


def tolerance(case):
    # Against 64 bits, over three seeds of the listed cases and 30 drawn ones:
    # up to 0.011 where the chains stay close -- 1e-7 to 7e-5 until a flipped
    # decision, and a flip moves one spin by up to its own size.  Chains too
    # long to stay close agree only where every update gives the same bits, as
    # the library's kernels do among one another.
    return {"rel": 0.03, "max": 0.99}


# ---------------------------------------------------------------------------
# The same chains in 64 bits
# ---------------------------------------------------------------------------

_W = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox-4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11) on int64 tensors
    holding 32-bit words; products wrap modulo 2^64, which keeps their words."""
    def words(m, a):
        p = a * m
        return (p >> 32) & _W, p & _W

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _W, (k1 + 0xBB67AE85) & _W
        h0, l0 = words(0xD2511F53, c0)
        h1, l1 = words(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return c0, c1, c2, c3


def _u(r):
    return ((r >> 9) * 2 + 1).double() * 2.0 ** -24


def _sphere(u0, u1):
    z = 2 * u0 - 1
    rho, phi = torch.sqrt(1 - z * z), 2 * math.pi * u1
    return torch.stack([rho * torch.cos(phi), rho * torch.sin(phi), z], -1)


def _keys(specs, replica=True):
    """Philox keys (B,1,1,1) of (seed, sample, replica) lists."""
    k0 = [s & _W for s, _, _ in specs]
    k1 = [(s >> 32) ^ ((2 * a + (r if replica else 0)) * 0x9E3779B9 & _W) for s, a, r in specs]
    return tuple(torch.tensor(k, dtype=torch.int64, device="cuda").view(-1, 1, 1, 1) for k in (k0, k1))


class _Chain:
    """A batch of lattices of one side, in 64 bits: s and J as (B, z, y, x, component)."""

    def __init__(self, L, specs, T, J=None):
        self.L, self.B = L, len(specs)
        n = torch.arange(L, device="cuda", dtype=torch.int64)
        x, y, z = n.view(1, 1, L), n.view(1, L, 1), n.view(L, 1, 1)
        self.site = (x + y * L + z * L * L).unsqueeze(0)
        self.colour = ((x + y + z) & 1).view(1, L, L, L, 1)
        self.key = _keys(specs)
        zero = torch.zeros((self.B, 1, 1, 1), dtype=torch.int64, device="cuda")
        r = _philox(self.site + zero, zero, zero + (1 << 24), zero, *self.key)
        self.s = _sphere(_u(r[0]), _u(r[1]))
        if J is None:  # Box & Muller from stream kind 2, under the key of replica 0, rounded to fp32
            r = _philox(self.site + zero, zero, zero + (2 << 24), zero, *_keys(specs, replica=False))
            u = [_u(a) for a in r]
            a, b = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
            J = torch.stack([a * torch.cos(2 * math.pi * u[1]), a * torch.sin(2 * math.pi * u[1]),
                             b * torch.cos(2 * math.pi * u[3])], -1).float()
        self.J = J.double().view(self.B, L, L, L, 3)
        self.beta = (1 / torch.tensor(T, dtype=torch.float64, device="cuda")).view(-1, 1, 1, 1)
        self.sweep = 0

    def field(self):
        h = 0
        for d, dim in ((0, 3), (1, 2), (2, 1)):
            j = self.J[..., d:d + 1]
            h = h + j * self.s.roll(-1, dim) + (j * self.s).roll(1, dim)
        return h

    def draw(self, kind, colour, hit):
        zero = torch.zeros((self.B, 1, 1, 1), dtype=torch.int64, device="cuda")
        return [_u(r) for r in _philox(self.site + zero, zero + self.sweep, zero + ((kind << 24) | (colour << 16) | hit),
                                       zero, *self.key)]

    @staticmethod
    def reflect(s, h):
        hh = (h * h).sum(-1, keepdim=True)
        t = 2 * (s * h).sum(-1, keepdim=True) / hh * h - s
        return torch.where(hh == 0, s, t)

    def metropolis(self, s, h, colour, hits, ball):
        for j in range(hits):
            u = self.draw(3, colour, j)
            p = _sphere(u[0], u[1])
            if ball:
                p = s + 0.5 * u[2].pow(1 / 3).unsqueeze(-1) * p
                p = p / p.norm(dim=-1, keepdim=True)
            de = -((p - s) * h).sum(-1)
            s = torch.where((u[3] < torch.exp(-self.beta * de)).unsqueeze(-1), p, s)
        return s

    def heatbath(self, h, colour):
        u = self.draw(4, colour, 0)
        hn = h.norm(dim=-1)
        x = self.beta * hn
        n = h / hn.unsqueeze(-1)
        sv = (-torch.log1p(u[0] * torch.expm1(-2 * x)) / x).clamp(0, 2)
        st = torch.sqrt(sv * (2 - sv))
        nx, ny, nz = n.unbind(-1)
        sign = torch.copysign(torch.ones_like(nz), nz)
        a = -1 / (sign + nz)
        b = nx * ny * a
        c1, c2 = st * torch.cos(2 * math.pi * u[1]), st * torch.sin(2 * math.pi * u[1])
        return (1 - sv).unsqueeze(-1) * n + torch.stack([
            c1 * (1 + sign * nx * nx * a) + c2 * b, c1 * sign * b + c2 * (sign + ny * ny * a),
            -c1 * sign * nx - c2 * ny], -1)

    def half(self, update, colour, hits=1, ball=False):
        h = self.field()
        if update == "or":
            t = self.reflect(self.s, h)
        elif update == "hb":
            t = self.heatbath(h, colour)
        else:
            t = self.metropolis(self.s, h, colour, hits, ball)
            if update == "met_or":
                t = self.reflect(t, h)
        self.s = torch.where(self.colour == colour, t, self.s)

    def run(self, case):
        for _ in range(case["sweeps"]):
            if case["update"] != "none":
                for c in (0, 1):
                    self.half(case["update"], c, case["hits"], case["proposal"] == "ball")
            for _ in range(case["n_or"]):
                for c in (0, 1):
                    self.half("or", c)
            self.sweep += 1
            if case["cadence"] and self.sweep % case["cadence"] == 0:
                self.s = self.s / self.s.norm(dim=-1, keepdim=True)

    def energy(self):
        e = 0
        for d, dim in ((0, 3), (1, 2), (2, 1)):
            e = e - (self.J[..., d] * (self.s * self.s.roll(-1, dim)).sum(-1)).sum((1, 2, 3))
        return e / self.L ** 3


def exact(case, seed):
    way, seed = case["way"], int(seed)
    if not _comparable(case):
        return None  # the chain in 64 bits is another one (or, served, too long)
    if way != "pool":
        c = _Chain(case["L"], [(seed, 1, 0)], [case["T"]], _couplings(case, seed))
        c.run(case)
        e = c.energy()
        return {"energy": e if way == "custom" else float(e), "spins": c.s.reshape(-1)}
    specs = _specs(case, seed)
    energies = torch.empty(len(specs), dtype=torch.float64)
    spins = [None] * len(specs)
    for L in _sides(case):
        at = [i for i, s in enumerate(specs) if s[0] == L]
        if not at:
            continue
        c = _Chain(L, [specs[i][1:4] for i in at], [specs[i][4] for i in at])
        c.run(case)
        for i, e, s in zip(at, c.energy().tolist(), c.s):
            energies[i], spins[i] = e, s.reshape(-1)
    return {"energies": energies.numpy(), "spins": torch.cat(spins)}
