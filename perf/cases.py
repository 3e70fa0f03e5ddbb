"""What this library is used for, as cases that can be timed: lattices of every size range and spin
encoding, annealing and sampling on sparse graphs, batches, and the serving queue, each through the entry
points that a program calls.  Sizes are those of the benchmark, the tests and the workload generators, or
lie in their ranges.

A case names a `kind`:
  lattice  one L x L context (INT8, PACKED or MULTISPIN): `mode` "step" runs n steps, "record" runs n steps
           with m and H of every step, "anneal" runs a schedule of n steps with best-energy tracking
  batch    groups of 32 replicas on lattices of mixed sizes stepped together: states in, n steps, states
           and observables out
  graph    one graph context (Erdos-Renyi, power-law, +-1 torus): "step" or "anneal"
  server   annealing jobs on Erdos-Renyi graphs through the serving queue, each job's result and final
           state fetched
"""
import math

import numpy as np
import torch

from paper_1904_06257_gb300 import shaken as S
from paper_1904_06257_gb300 import workloads as W

ENCODINGS = {"int8": S.INT8, "packed": S.PACKED, "multispin": S.MULTISPIN}
GROUP_SIDES = (32, 64, 128, 256, 512)


def listed():
    return [
        # The smallest use: one small lattice watched step by step (m and H of every step).
        dict(name="lattice64_record", kind="lattice", enc="int8", L=64, R=1, n=500, mode="record",
             J=1.0, q=1.0, lam=0.0, beta=0.40, boundary=0),
        # Metastability curves: replicas of one small lattice, m and H of every step, q < lambda < J.
        dict(name="multispin64_record", kind="lattice", enc="multispin", L=64, R=128, n=200, mode="record",
             J=1.0, q=0.1, lam=0.15, beta=1.3, boundary=0),
        # The batched workload: 128 groups of 32 replicas, states uploaded, 20 steps, states and
        # observables back.
        dict(name="multispin_batch", kind="batch", groups=128, n=20, J=1.0, q=1.0, lam=0.0,
             beta_lo=0.3, beta_hi=0.6),
        # One plain lattice near criticality, measured every 100 steps.
        dict(name="lattice4096_int8", kind="lattice", enc="int8", L=4096, R=1, n=100, mode="step",
             J=1.0, q=1.0, lam=0.0, beta=0.4407, boundary=0),
        # The same sweep's points with a field and q != J, packed, on a side that is no power of two.
        dict(name="lattice2912_packed_field", kind="lattice", enc="packed", L=2912, R=1, n=100, mode="step",
             J=1.0, q=0.5, lam=0.01, beta=0.48, boundary=0),
        # The largest single lattice of the tests: 2^28 sites, one byte each.
        dict(name="lattice16384_int8", kind="lattice", enc="int8", L=16384, R=1, n=12, mode="step",
             J=1.0, q=1.0, lam=0.0, beta=0.4407, boundary=0),
        # A small annealing job: one word of replicas on a sparse graph, thousands of short half steps.
        dict(name="graph2e3_anneal", kind="graph", graph="er", n=2000, degree=6.0, R=32, steps=500,
             mode="anneal", real=False, q=1.0, field=0.0, beta=1.0, ladder=False),
        # Annealing +-1 couplings on a large random graph (max-cut), best energy of every step.
        dict(name="graph1e6_anneal", kind="graph", graph="er", n=1_000_000, degree=8.0, R=256, steps=20,
             mode="anneal", real=False, q=1.0, field=0.0, beta=1.0, ladder=False),
        # Gaussian couplings and random fields on the same graph, sampling at one temperature.
        dict(name="graph1e6_real", kind="graph", graph="er", n=1_000_000, degree=8.0, R=256, steps=10,
             mode="step", real=True, q=1.0, field=0.1, beta=1.0, ladder=False),
        # A hub-heavy graph: power-law degrees, +-1 couplings, random fields.
        dict(name="powerlaw1e6_step", kind="graph", graph="powerlaw", n=1_000_000, degree=8.0, R=256,
             steps=10, mode="step", real=False, q=1.0, field=0.1, beta=1.0, ladder=False),
        # The 2D Edwards-Anderson anneal: +-1 torus of side 256, q > 2.
        dict(name="ea256_anneal", kind="graph", graph="torus", n=65536, degree=4.0, R=256, steps=100,
             mode="anneal", real=False, q=2.5, field=0.0, beta=1.0, ladder=False),
        # Serving: a handful of jobs of mixed sizes through the queue.
        dict(name="server_jobs", kind="server", jobs=6, n_lo=1000, n_hi=30000, r_hi=256, steps=300),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ones' ranges."""
    kind = rng.choice(["small", "record", "batch", "single", "single", "replicas", "graph", "graph",
                       "graph_small", "real", "server"])
    fields = dict(J=1.0, q=rng.choice([0.5, 1.0, 1.0, 2.0, 4.0]), lam=rng.choice([0.0, 0.0, 0.01, 0.15]),
                  beta=rng.choice([0.40, 0.4407, 0.48, 0.7]), boundary=rng.choice([0, 0, 0, 1]))
    if kind == "small":  # INT8 / PACKED, whole run in one launch
        return dict(kind="lattice", enc=rng.choice(["int8", "packed"]), L=32 * rng.randint(1, 11),
                    R=rng.choice([1, 1, 3, 16]), n=rng.randint(50, 600),
                    mode=rng.choice(["record", "step", "anneal"]), **fields)
    if kind == "record":
        return dict(kind="lattice", enc="multispin", L=32 * rng.randint(1, 6), R=32 * rng.randint(1, 8),
                    n=rng.randint(30, 250), mode=rng.choice(["record", "step", "anneal"]), **fields)
    if kind == "batch":
        return dict(kind="batch", groups=int(_log(rng, 3, 128)), n=rng.randint(5, 40), J=1.0,
                    q=rng.choice([0.5, 1.0, 1.0, 2.0]), lam=rng.choice([0.0, 0.0, 0.01]), beta_lo=0.3,
                    beta_hi=rng.uniform(0.35, 0.7))
    if kind == "single":  # one lattice beyond one block's shared memory
        L = 32 * int(_log(rng, 12, 512))
        return dict(kind="lattice", enc=rng.choice(["int8", "packed"]), L=L, R=1,
                    n=max(9, min(200, int(1.5e9 / (L * L)))), mode="step", **fields)
    if kind == "replicas":  # several replicas of a mid-size lattice
        L = 32 * int(_log(rng, 12, 64))
        return dict(kind="lattice", enc=rng.choice(["int8", "packed", "multispin"]), L=L,
                    R=32 * rng.randint(1, 2), n=rng.randint(6, 12), mode=rng.choice(["step", "anneal"]),
                    **fields)
    q = rng.choice([0.7, 1.0, 1.0, 2.5])
    if kind == "graph":
        graph = rng.choice(["er", "er", "powerlaw", "torus"])
        R = 32 * rng.choice([1, 2, 3, 5, 8, 12])
        n = int(_log(rng, 2e4, min(8e5, 1.6e8 / R)))
        n = int(math.isqrt(n)) ** 2 if graph == "torus" else n
        mode = rng.choice(["anneal", "step"])
        # annealing jobs carry no field, sampling runs may; a ladder: one temperature per replica
        return dict(kind="graph", graph=graph, n=n, degree=4.0 if graph == "torus" else rng.uniform(3, 16),
                    R=R, steps=rng.randint(4, 20), mode=mode, real=False,
                    q=q, field=0.0 if mode == "anneal" else rng.choice([0.0, 0.1]), beta=1.0,
                    ladder=mode == "step" and rng.random() < 0.25)
    if kind == "graph_small":
        return dict(kind="graph", graph="er", n=int(_log(rng, 1e3, 2e4)), degree=rng.uniform(3, 16),
                    R=32 * rng.choice([1, 2, 4]), steps=rng.randint(50, 400), mode="anneal", real=False, q=q,
                    field=0.0, beta=1.0, ladder=False)
    if kind == "real":
        return dict(kind="graph", graph="er", n=int(_log(rng, 2e3, 6e5)), degree=rng.uniform(3, 16),
                    R=32 * rng.choice([1, 2, 5, 8]), steps=rng.randint(4, 15), mode="step", real=True, q=q,
                    field=rng.choice([0.0, 0.1]), beta=rng.uniform(0.5, 2.0), ladder=False)
    return dict(kind="server", jobs=rng.randint(2, 8), n_lo=1000, n_hi=int(_log(rng, 3e3, 3e4)),
                r_hi=rng.choice([64, 128, 256]), steps=rng.randint(100, 400))


# ------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _edges(case, seed):
    """Edge arrays u, v (host int32) of the case's graph."""
    g, n = _gen(seed), case["n"]
    if case["graph"] == "torus":
        return W.lattice_as_graph(math.isqrt(n))
    m = int(n * case["degree"] / 2)
    if case["graph"] == "powerlaw":  # both ends in proportion to (i + 1)^(-1 / 1.1): exponent 2.1
        w = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** (-1.0 / 1.1)
        c = torch.cumsum(w, 0)
        p = torch.rand(2, m, device="cuda", dtype=torch.float64, generator=g) * c[-1]
        ends = torch.searchsorted(c, p).clamp_(max=n - 1)
    else:
        ends = torch.randint(n, (2, m), device="cuda", generator=g)
    a, b = ends.min(0).values, ends.max(0).values
    key = torch.unique((a * n + b)[a != b])
    return (key // n).to(torch.int32).cpu().numpy(), (key % n).to(torch.int32).cpu().numpy()


def _couplings(case, seed, m):
    g = _gen(seed + 1)
    if case.get("real"):
        return torch.randn(m, device="cuda", generator=g).cpu().numpy()
    return (1.0 - 2.0 * torch.randint(2, (m,), device="cuda", generator=g)).to(torch.float32).cpu().numpy()


def _schedule(n):
    return W.linear_schedule(0.1, 3.0, n)


def _sides(case, seed):
    """Every side equally often (up to the remainder), in an order of the seed."""
    sides = [GROUP_SIDES[-1 - k % len(GROUP_SIDES)] for k in range(case["groups"])]
    return [sides[k] for k in np.random.default_rng(seed).permutation(len(sides))]


def _group_betas(case):
    return W.beta_grid(32 * case["groups"], case["beta_lo"], case["beta_hi"], 64)


def _random_bytes(nbytes, seed):
    x = torch.randint(-2**31, 2**31, (nbytes // 4,), device="cuda", generator=_gen(seed + 2)).to(torch.int32)
    return x.cpu().view(torch.uint8).pin_memory()


def _graph_betas(case):
    return np.linspace(0.2, 2.0, case["R"]) if case["ladder"] else case["beta"]


def _jobs(case):
    """The jobs of a serving case: sizes and replicas spread over the logarithm of their ranges, degrees
    and steps over theirs, in different orders."""
    k = case["jobs"]
    at = [(i + 0.5) / k for i in range(k)]
    step = next(s for s in (3, 5, 7, 11) if math.gcd(s, k) == 1)
    jobs = []
    for i, x in enumerate(at):
        y, z = at[(i * step + 1) % k], at[(i * step + k // 2) % k]
        jobs.append(dict(graph="er", n=int(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** x), degree=3.0 + 13.0 * y,
                         R=32 * round((case["r_hi"] / 32) ** z), steps=int(case["steps"] * (0.5 + 0.5 * y))))
    return jobs


class _State:
    """Handles of one case; released with the object."""

    def __init__(self, case, seed):
        self.case, self.seed, self.ctxs, self.batch, self.server = case, seed, [], None, None

    def __del__(self):
        if self.server is not None:
            S.shaken_server_free(self.server)
        for c in self.ctxs:
            S.shaken_free(c)
        if self.batch is not None:
            S.shaken_batch_free(self.batch)


def _pinned(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8).pin_memory()


def prepare(case, seed):
    st = _State(case, seed)
    if case["kind"] == "lattice":
        p = S.Problem(S.LATTICE, ENCODINGS[case["enc"]], case["R"], case["beta"], case["q"], L=case["L"],
                      J=case["J"], lambda_const=case["lam"], boundary=case["boundary"])
        st.ctxs.append(S.shaken_init(p, seed))
        st.schedule = _schedule(case["n"])
        st.out = _pinned(S.shaken_state_bytes(st.ctxs[0]))
    elif case["kind"] == "batch":
        betas, st.batch = _group_betas(case), S.shaken_batch_create()
        for g, L in enumerate(_sides(case, seed)):
            p = S.Problem(S.LATTICE, S.MULTISPIN, 32, betas[32 * g:32 * g + 32], case["q"], L=L, J=case["J"],
                          lambda_const=case["lam"])
            st.ctxs.append(S.shaken_init(p, seed + g))
            S.shaken_batch_add(st.batch, st.ctxs[-1])
        st.bytes = S.shaken_batch_state_bytes(st.batch)
        st.inp, st.out = _random_bytes(st.bytes, seed), _pinned(st.bytes)
    elif case["kind"] == "graph":
        u, v = _edges(case, seed)
        lam = W.fields_normal(case["n"], case["field"], seed) if case["field"] else None
        p = S.Problem(S.GRAPH, S.MULTISPIN, case["R"], _graph_betas(case), case["q"], n=case["n"], u=u, v=v,
                      J_edge=_couplings(case, seed, u.size), J_is_integer=not case["real"], lambda_=lam,
                      orientation=S.ORIENT_GIVEN if case["graph"] == "torus" else S.ORIENT_MIN_MAX)
        st.ctxs.append(S.shaken_init(p, seed))
        st.schedule = _schedule(case["steps"])
        st.out = _pinned(S.shaken_state_bytes(st.ctxs[0]))
    else:
        st.server = S.shaken_server_create(8 << 30, 64)
        S.shaken_server_set_policy(st.server, 3e8, 0, True)
        st.jobs = []
        for k, j in enumerate(_jobs(case)):
            u, v = _edges(j, seed + 10 * k)
            p = S.Problem(S.GRAPH, S.MULTISPIN, j["R"], 0.1, 1.0, n=j["n"], u=u, v=v,
                          J_edge=_couplings(j, seed + 10 * k, u.size), J_is_integer=True)
            st.jobs.append((p, seed + k, _schedule(j["steps"]), j["n"] * j["R"] // 8))
    return st


def _fields(obs):
    return {f: obs[f] for f in ("magnetization", "energy", "pair_energy", "best_energy", "best_step",
                                "cut_edges", "cut_weight")}


def run(st):
    case = st.case
    if case["kind"] == "lattice":
        c, out = st.ctxs[0], {}
        if case["mode"] == "record":
            out["m"], out["H"] = S.shaken_step_record(c, case["n"], case["R"])
        elif case["mode"] == "anneal":
            S.shaken_anneal(c, st.schedule)
        else:
            S.shaken_step(c, case["n"])
        S.shaken_get_state_raw_async(c, st.out.data_ptr(), st.out.numel())
        out.update(_fields(S.shaken_observables(c, case["R"])))
        return {"state": st.out, **out}
    if case["kind"] == "batch":
        S.shaken_batch_set_states_raw(st.batch, st.inp.data_ptr(), st.bytes)
        S.shaken_batch_step(st.batch, case["n"])
        S.shaken_batch_get_states_raw_async(st.batch, st.out.data_ptr(), st.bytes)
        return {"state": st.out, **_fields(S.shaken_batch_observables(st.batch, 32 * case["groups"]))}
    if case["kind"] == "graph":
        c = st.ctxs[0]
        if case["mode"] == "anneal":
            S.shaken_anneal(c, st.schedule)
        else:
            S.shaken_step(c, case["steps"])
        S.shaken_get_state_raw_async(c, st.out.data_ptr(), st.out.numel())
        return {"state": st.out, **_fields(S.shaken_observables(c, case["R"]))}
    ids = [S.shaken_server_submit(st.server, p, seed, sched) for p, seed, sched, _ in st.jobs]
    S.shaken_server_drain(st.server, 60.0)
    out = {}
    for k, (jid, (p, _, _, nbytes)) in enumerate(zip(ids, st.jobs)):
        out["obs%d" % k] = _fields(S.shaken_server_result(st.server, jid, p.replicas)[0])["best_energy"]
        out["state%d" % k] = S.shaken_server_result_state(st.server, jid, nbytes)
    return out


# ------------------------------------------------------------------------------------------ work
def _lattice_state(case):
    N = case["L"] * case["L"]
    return N * case["R"] if case["enc"] == "int8" else N * case["R"] // 8


def work(case):
    """Bytes: the state in and out once, the graph once, the results.  Operations: per 32 decisions two
    Philox calls (20 products and 20 xors each) and eight planes compared in four operations, plus the
    neighbours' contribution (lattice: 4; graph: one operation per edge and word); real couplings: eight
    calls per 32 draws, an addition per edge and ten operations per decision."""
    if case["kind"] == "lattice":
        N, s = case["L"] ** 2, _lattice_state(case)
        out = 56 * case["R"] + (16 * case["R"] * case["n"] if case["mode"] == "record" else 0)
        return {"bytes": 2 * s + out, "flops": 2.0 * case["n"] * N * case["R"] * 116 / 32}
    if case["kind"] == "batch":
        N = sum(x * x for x in _sides(case, 0))
        return {"bytes": 8 * N + 56 * 32 * case["groups"], "flops": 2.0 * case["n"] * N * 116}
    if case["kind"] == "graph":
        n, m, R = case["n"], case["n"] * case["degree"] / 2, case["R"]
        if case["real"]:
            ops = 2.0 * case["steps"] * R * (20 * n + m)
        else:
            ops = 2.0 * case["steps"] * (R / 32) * (112 * n + m)
        return {"bytes": 2 * n * R / 8 + m * (16 if case["real"] else 8) + 8 * n, "flops": ops}
    jobs = [(j, j["n"] * j["degree"] / 2) for j in _jobs(case)]
    return {"bytes": sum(j["n"] * j["R"] / 8 + 12 * m for j, m in jobs),
            "flops": sum(2.0 * j["steps"] * (j["R"] / 32) * (112 * j["n"] + m) for j, m in jobs)}


# ------------------------------------------------------------------------------------------ exact values
_MASK = 0xFFFFFFFF


def _philox(seed, a, b, t, c3):
    """Philox-4x32-10 on int64 tensors of 32-bit words: the four output words."""
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    c = [a, b + torch.zeros_like(a), torch.full_like(a, t), torch.full_like(a, c3)]
    for r in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & _MASK) ^ c[1] ^ ((k0 + r * 0x9E3779B9) & _MASK), p1 & _MASK,
             ((p0 >> 32) & _MASK) ^ c[3] ^ ((k1 + r * 0xBB67AE85) & _MASK), p0 & _MASK]
    return c


def _plane_draws(seed, a, b, t, half):
    """The 32 draws of every lane word, from its 32 plane words: [..., 32]."""
    k = torch.arange(32, device="cuda")
    u = torch.zeros(a.shape + (32,), dtype=torch.int64, device="cuda")
    for c in range(8):
        for i, w in enumerate(_philox(seed, a, b, t, half + 2 * c)):
            u += ((w[..., None] >> k) & 1) << (31 - 4 * c - i)
    return u


def _threshold(h, beta):
    return torch.floor(2.0**32 / (1.0 + torch.exp(-2.0 * beta * h)))


def _pack(bits):
    """Lanes [..., 32] of 0 / 1 -> little-endian bytes."""
    w = (bits.to(torch.int64) << torch.arange(32, device="cuda")).sum(-1)
    return torch.stack([(w >> s) & 255 for s in (0, 8, 16, 24)], -1).to(torch.uint8).reshape(-1).cpu()


class _Lattice:
    """An L x L torus: spins s [jobs, L, L, 32 lanes] (multispin) or [replicas, L, L], +-1 in 64 bits."""

    def __init__(self, enc, L, R, J, q, lam, beta, seed, boundary=0):
        self.enc, self.L, self.R, self.J, self.q, self.lam, self.seed = enc, L, R, J, q, lam, seed
        self.multi = enc == "multispin"
        jobs, words = (R // 32, L * L) if self.multi else (R, L * L // 32)
        self.a = torch.arange(words, device="cuda").expand(jobs, words)
        self.b = torch.arange(jobs, device="cuda")[:, None]
        self.shape = (jobs, L, L, 32) if self.multi else (jobs, L, L)
        b = torch.as_tensor(np.broadcast_to(np.asarray(beta, np.float64), (R,)).copy(), device="cuda")
        self.beta = b.reshape(jobs, 1, 1, 32) if self.multi else b.reshape(jobs, 1, 1)
        self.frozen = torch.zeros(self.shape, dtype=torch.bool, device="cuda")
        if boundary:
            self.frozen[:, 0], self.frozen[:, :, 0] = True, True
        first = _philox(seed, self.a, self.b, _MASK, 0)[0]
        up = ((first[..., None] >> torch.arange(32, device="cuda")) & 1) == 0
        self.s = self._spins(up)
        self.prime, self.t = self.s, 0

    def _spins(self, up):
        s = torch.where(up.reshape(self.shape), 1.0, -1.0).double()
        return torch.where(self.frozen, 1.0, s)

    def half(self, s, half, beta):
        d = 1 if half == 0 else -1  # dl reads row i - 1 and column j - 1, ur the opposite ones
        h = self.J * (s.roll(d, 1) + s.roll(d, 2)) + self.q * s + self.lam
        u = _plane_draws(self.seed, self.a, self.b, self.t, half).reshape(self.shape)
        return self._spins(u < _threshold(h, beta))

    def step(self, beta=None):
        beta = self.beta if beta is None else beta
        self.prime = self.half(self.s, 0, beta)
        self.s = self.half(self.prime, 1, beta)
        self.t += 1

    def _sum(self, x):
        return x.sum((1, 2)).reshape(-1)

    def energy(self):
        s = self.s
        M, E = self._sum(s), self._sum(s * (s.roll(1, 1) + s.roll(1, 2)))
        return M, E, -(self.J * E) - 2.0 * self.lam * M

    def observables(self, best, best_step):
        s, p, N = self.s, self.prime, self.L * self.L
        M, E, H = self.energy()
        P1, P2 = self._sum(s * (p.roll(-1, 1) + p.roll(-1, 2))), self._sum(s * p)
        cut = (2 * N - E) / 2
        better = H < best
        return {"magnetization": M / N, "energy": H,
                "pair_energy": -(self.J * P1 + self.q * P2 + self.lam * (M + self._sum(p))),
                "best_energy": torch.where(better, H, best),
                "best_step": torch.where(better, torch.full_like(best_step, self.t), best_step),
                "cut_edges": cut.to(torch.int64), "cut_weight": -self.J * cut}

    def state(self):
        if self.enc == "int8":
            return self.s.to(torch.int8).reshape(-1).view(torch.uint8).cpu()
        return _pack((self.s > 0).reshape(-1, 32))


def _host(d):
    return {k: v.cpu().numpy() if isinstance(v, torch.Tensor) and k != "state" else v for k, v in d.items()}


def _exact_lattice(case, seed):
    x = _Lattice(case["enc"], case["L"], case["R"], case["J"], case["q"], case["lam"], case["beta"], seed,
                 case["boundary"])
    best = torch.full((case["R"],), math.inf, dtype=torch.float64, device="cuda")
    best_step = torch.full((case["R"],), -1, dtype=torch.int64, device="cuda")
    m, Hs, sched = [], [], _schedule(case["n"])
    for k in range(case["n"]):
        if case["mode"] != "step":
            M, _, H = x.energy()
            m.append(M / (x.L * x.L))
            Hs.append(H)
            best_step = torch.where(H < best, torch.full_like(best_step, k), best_step)
            best = torch.minimum(best, H)
        x.step(float(sched[k]) if case["mode"] == "anneal" else None)
    out = {"state": x.state(), **x.observables(best, best_step)}
    if case["mode"] == "record":
        out.update(m=torch.stack(m), H=torch.stack(Hs))
    return _host(out)


def _exact_batch(case, seed):
    sides, betas = _sides(case, seed), _group_betas(case)
    words = _random_bytes(sum(4 * L * L for L in sides), seed).view(torch.int32).cuda().to(torch.int64) & _MASK
    at, parts = 0, []
    for g, L in enumerate(sides):
        x = _Lattice("multispin", L, 32, case["J"], case["q"], case["lam"], betas[32 * g:32 * g + 32], seed + g)
        w = words[at:at + L * L]
        at += L * L
        x.s = x.prime = x._spins(((w[:, None] >> torch.arange(32, device="cuda")) & 1) == 1)
        for _ in range(case["n"]):
            x.step()
        inf = torch.full((32,), math.inf, dtype=torch.float64, device="cuda")
        parts.append({"state": x.state(), **x.observables(inf, torch.zeros(32, dtype=torch.int64, device="cuda"))})
    return _host({k: torch.cat([p[k] for p in parts]) for k in parts[0]})


def _exact_graph(case, seed):
    """+-1 couplings: spins [n, R] in 64 bits."""
    n, R, dev = case["n"], case["R"], "cuda"
    uh, vh = _edges(case, seed)
    Jh = _couplings(case, seed, uh.size)
    a, b = (uh, vh) if case["graph"] == "torus" else (np.minimum(uh, vh), np.maximum(uh, vh))
    tail, head = torch.as_tensor(a, device=dev).long(), torch.as_tensor(b, device=dev).long()
    J = torch.as_tensor(Jh, device=dev).double()[:, None]
    lam = (torch.as_tensor(W.fields_normal(n, case["field"], seed), device=dev).double()[:, None] if case["field"]
           else torch.zeros(n, 1, dtype=torch.float64, device=dev))
    beta0 = torch.as_tensor(np.broadcast_to(np.asarray(_graph_betas(case), np.float64), (R,)).copy(), device=dev)
    x = torch.arange(n, device=dev)[:, None].expand(n, R // 32)
    g = torch.arange(R // 32, device=dev)[None, :]
    words = [w for c in range(8) for w in _philox(seed, x, g, _MASK, 2 * c)]
    s = torch.where(torch.stack(words, -1) < 2**31, 1.0, -1.0).double().reshape(n, R)
    prime, sched = s, _schedule(case["steps"])
    best = torch.full((R,), math.inf, dtype=torch.float64, device=dev)
    best_step = torch.full((R,), -1, dtype=torch.int64, device=dev)

    def total(x, y):
        return (J * x[tail] * y[head]).sum(0)

    def half(s, half, t, beta):
        src, dst = (tail, head) if half == 0 else (head, tail)
        h = torch.zeros_like(s).index_add_(0, dst, J * s[src]) + case["q"] * s + lam
        u = _plane_draws(seed, x, g, t, half).reshape(n, R)
        return torch.where(u < _threshold(h, beta), 1.0, -1.0).double()

    for t in range(case["steps"]):
        beta = beta0
        if case["mode"] == "anneal":
            beta = float(sched[t])
            H = -total(s, s) - 2.0 * (lam * s).sum(0)
            best_step = torch.where(H < best, torch.full_like(best_step, t), best_step)
            best = torch.minimum(best, H)
        prime = half(s, 0, t, beta)
        s = half(prime, 1, t, beta)
    E, LS = total(s, s), (lam * s).sum(0)
    H, better = -E - 2.0 * LS, -E - 2.0 * LS < best
    return _host({
        "state": _pack((s > 0).reshape(n, R // 32, 32)), "magnetization": s.sum(0) / n, "energy": H,
        "pair_energy": -(total(s, prime) + case["q"] * (s * prime).sum(0) + LS + (lam * prime).sum(0)),
        "best_energy": torch.where(better, H, best),
        "best_step": torch.where(better, torch.full_like(best_step, case["steps"]), best_step),
        "cut_edges": (s[tail] != s[head]).sum(0), "cut_weight": 0.5 * (E - J.sum())})


def exact(case, seed):
    """The chain itself in plain 64-bit torch; None where that would take long, or where the decisions are
    those of 32-bit field sums (real couplings)."""
    if case["kind"] == "lattice":
        sites = case["L"] ** 2 * case["R"]
        return _exact_lattice(case, seed) if sites <= 2**25 and case["n"] * sites <= 2e9 else None
    if case["kind"] == "batch":
        return _exact_batch(case, seed) if case["n"] * case["groups"] <= 300 else None
    if case["kind"] == "graph" and not case["real"]:
        sites = case["n"] * case["R"]
        return _exact_graph(case, seed) if sites <= 2**25 and case["steps"] * sites <= 2e9 else None
    return None
