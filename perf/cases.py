"""Work that users of this package have it do, at fixed sizes, for timing and for comparing results.

listed() names the cases, draw() gives further ones of the same ranges, prepare() makes what a
program holds before the call, run() is the call and work() what it cannot do without.  exact()
restates the Ant System and the MAX-MIN Ant System in plain torch for the pheromone in 64 bits.

Kinds of case:
  solve   one instance from the host and back: create, options, iterate, best tour, pheromone
  step    one iteration of a handle that is kept, and its best tour so far
  pool    a group of requests through a kept pool: admit, step until done, results, release
  update  the allocation-free pheromone update on device arrays
"""
import math

import numpy as np
import torch

from paper_1101_2678_gb300 import aco, instances

SELECTION = {"eq1": aco.ACO_SELECT_EQ1, "data-parallel": aco.ACO_SELECT_DATA_PARALLEL,
             "exp-race": aco.ACO_SELECT_EXP_RACE}
RULES = {"as": (1.0, 2.0, 0.5), "mmas": (1.0, 2.0, 0.02), "acs": (1.0, 2.0, 0.1)}  # alpha, beta, rho
P_BEST = 0.05
Q0, XI = 0.9, 0.1


def solve(n, m, iterations, rule="as", selection="eq1", nn=0, clustered=False, coords=False, **name):
    return dict(kind="solve", n=n, m=m, iterations=iterations, rule=rule, selection=selection, nn=nn,
                clustered=clustered, coords=coords, **name)


def listed():
    return [
        # The paper's smallest instance size, a whole run: a step's latency and the launches count.
        solve(48, 48, 100, name="as n48"),
        # The paper's middle size, m = n, from a distance matrix.
        solve(1002, 1002, 20, name="as n1002"),
        # The paper's largest size, m = n, clustered: the default benchmark workload.
        solve(2392, 2392, 10, clustered=True, name="as n2392"),
        # The largest request a server takes: n = 4096 coordinates, m = 1024 ants.
        solve(4096, 1024, 5, coords=True, name="as n4096 m1024"),
        # MAX-MIN Ant System at an odd middle size.
        solve(517, 517, 40, rule="mmas", name="mmas n517"),
        # Candidate lists, as large instances are solved in practice.
        solve(2392, 2392, 10, nn=30, clustered=True, coords=True, name="as n2392 nn30"),
        # The Ant Colony System with its usual ten ants.
        solve(1002, 10, 10, rule="acs", name="acs n1002 m10"),
        # The paper's own data-parallel selection rule.
        solve(1002, 1002, 20, selection="data-parallel", name="data-parallel n1002"),
        # Eq. 1 by a race of exponentials, one random number per candidate.
        solve(1002, 1002, 5, selection="exp-race", name="exp-race n1002"),
        # A server's group of requests of many sizes, side by side in one pool.
        dict(kind="pool", count=28, lo=48, hi=1024, sizes=4, iterations=30, name="pool 28 requests"),
        # A caller that looks at the best tour after every iteration.
        dict(kind="step", n=48, m=48, rule="mmas", name="mmas n48 step"),
        # The update alone, on arrays of a program that may not allocate.
        dict(kind="update", n=1002, m=1002, name="update n1002"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    if pick < 0.08:
        return dict(kind="step", n=_log_uniform(rng, 24, 300), m=rng.randint(24, 96), rule="mmas")
    if pick < 0.16:
        return dict(kind="update", n=_log_uniform(rng, 48, 1024), m=_log_uniform(rng, 48, 2048))
    if pick < 0.28:
        return dict(kind="pool", count=rng.randint(8, 28), lo=48, hi=_log_uniform(rng, 300, 1024),
                    sizes=rng.randint(1, 1 << 20), iterations=rng.randint(10, 25))
    way = rng.choice(["as", "as", "as", "as", "mmas", "mmas", "nn", "nn", "acs", "data-parallel",
                      "exp-race"])
    n = _log_uniform(rng, 48, 1500 if way in ("data-parallel", "exp-race") else 4096)
    m = 10 if way == "acs" else rng.choice([n, min(n, 1024), rng.randint(max(n // 4, 1), n)])
    # microseconds of an iteration, roughly: keeps a drawn case below the largest listed ones
    us = {"acs": 5.0 * n, "nn": n * (0.8 + m / 3000),
          "exp-race": n * (2 + m * n / 2.5e5)}.get(way, n * (1 + m * n / 2e6))
    return solve(n, m, max(1, min(60, int(25000 / us))), rule=way if way in RULES else "as",
                 selection=way if way in SELECTION else "eq1", nn=rng.randint(15, 32) if way == "nn" else 0,
                 clustered=rng.random() < 0.5, coords=n > 2500 or rng.random() < 0.3)


def _instance(n, seed, clustered=False):
    if clustered:
        return instances.clustered_instance(n, seed)
    return instances.uniform_instance(n, 1000 if n < 500 else 10000, seed)


def _handle(case, inst, seed):
    """A handle with the case's rule and options, as a program sets it up."""
    alpha, beta, rho = RULES[case["rule"]]
    if case.get("coords"):
        h = aco.aco_create_coords(inst.coords, alpha, beta, rho, case["m"], seed)
    else:
        h = aco.aco_create(inst.dist, alpha, beta, rho, case["m"], seed)
    if case["rule"] == "mmas":
        aco.aco_set_mmas(h, P_BEST, False)
    elif case["rule"] == "acs":
        aco.aco_set_acs(h, Q0, XI)
    if case.get("nn"):
        aco.aco_set_option(h, aco.ACO_OPT_NN_LIST, case["nn"])
    if case.get("selection", "eq1") != "eq1":
        aco.aco_set_option(h, aco.ACO_OPT_SELECTION, SELECTION[case["selection"]])
    return h


def _sizes(case):
    """City counts of a pool's requests."""
    return instances.log_uniform_sizes(case["count"], case["lo"], case["hi"], case["sizes"])


class _Kept:
    """A handle or pool that is given back with its owner."""

    def __init__(self, handle, destroy):
        self.handle, self.destroy = handle, destroy

    def __del__(self):
        self.destroy(self.handle)


def _update_arrays(case, seed):
    """Tours like those of a converging colony (segments of one tour reversed), their lengths,
    eta^beta and a pheromone matrix, on the device."""
    n, m = case["n"], case["m"]
    rng = np.random.default_rng(seed)
    dist = _instance(n, seed).dist
    base, left = [0], np.ones(n, bool)
    for _ in range(n - 1):
        left[base[-1]] = False
        base.append(int(np.argmin(np.where(left, dist[base[-1]], 1 << 30))))
    tours = np.tile(np.array(base, np.int32), (m, 1))
    for t in tours:
        for a, b in np.sort(rng.integers(0, n, (8, 2)), axis=1):
            t[a:b] = t[a:b][::-1].copy()
    tours = np.concatenate([tours, tours[:, :1]], axis=1)
    lens = dist[tours[:, :-1], tours[:, 1:]].sum(1, dtype=np.int64)
    heta = np.zeros((n, n), np.float32)
    off = ~np.eye(n, dtype=bool)
    heta[off] = (1.0 / dist[off].astype(np.float64) ** 2).astype(np.float32)
    u = np.triu(rng.uniform(0.1, 2.0, (n, n)) * m / float(lens.min()), 1)
    tau = (u + u.T).astype(np.float32)
    return {"tours": tours, "lens": lens, "heta": heta, "tau": tau}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        inst = _instance(case["n"], seed, case["clustered"])
        if not case["coords"]:
            inst.dist  # built once, on first use
        return dict(case=case, inst=inst, seed=seed)
    if kind == "step":
        h = _handle(case, _instance(case["n"], seed), seed)
        return dict(case=case, kept=_Kept(h, aco.aco_destroy))
    if kind == "pool":
        insts = [_instance(int(n), seed + i, i % 2 == 1) for i, n in enumerate(_sizes(case))]
        room = sum(aco.aco_pool_bytes_needed(i.n, i.n) for i in insts)
        state = dict(case=case, insts=insts, seed=seed,
                     kept=_Kept(aco.aco_pool_create(case["count"], room), aco.aco_pool_destroy))
        slots = _admit(state, 1)  # a server tunes its pool before it takes requests
        aco.aco_pool_autotune(state["kept"].handle)
        for s in slots:
            aco.aco_pool_release(state["kept"].handle, s)
        return state
    arrays = {k: torch.from_numpy(v).cuda() for k, v in _update_arrays(case, seed).items()}
    return dict(case=case, choice=torch.empty_like(arrays["heta"]), **arrays)


def _admit(state, iterations):
    p = state["kept"].handle
    alpha, beta, rho = RULES["as"]
    return [aco.aco_pool_admit_coords(p, inst.coords, alpha, beta, rho, inst.n, state["seed"] + i,
                                      iterations) for i, inst in enumerate(state["insts"])]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        n = case["n"]
        h = _handle(case, state["inst"], state["seed"])
        try:
            aco.aco_iterate(h, case["iterations"])
            tour, length = aco.aco_best_tour(h, n)
            return dict(tour=tour, length=length, tau=aco.aco_get_pheromone(h, n))
        finally:
            aco.aco_destroy(h)
    if kind == "step":
        h, n = state["kept"].handle, case["n"]
        aco.aco_iterate(h, 1)
        tour, length = aco.aco_best_tour(h, n)
        return dict(tour=tour, length=length, tau=aco.aco_get_pheromone(h, n))
    if kind == "pool":
        p, insts = state["kept"].handle, state["insts"]
        slots = _admit(state, case["iterations"])
        while aco.aco_pool_step(p):
            pass
        found = [aco.aco_pool_result(p, s, i.n) for s, i in zip(slots, insts)]
        taus = [aco.aco_pool_pheromone(p, s, i.n) for s, i in zip(slots, insts)]
        for s in slots:
            aco.aco_pool_release(p, s)
        return dict(tours=[t for t, _ in found], tau=taus,
                    lengths=np.array([c for _, c in found], np.int64))
    aco.aco_update_pheromone_noalloc(
        case["n"], case["m"], *(state[k].data_ptr() for k in ("tours", "lens", "heta", "tau", "choice")),
        1.0, RULES["as"][2], torch.cuda.current_stream().cuda_stream)
    return dict(tau=state["tau"], choice=state["choice"])


def work(case):
    """Bytes: the instance in, pheromone and tour out.  Operations: for every ant and step one
    multiplication-free look at each candidate (a sum and a comparison), and the update's cells."""
    kind = case["kind"]
    if kind == "pool":
        ns = [int(n) for n in _sizes(case)]
        return dict(bytes=sum(8 * n + 4 * n * n + 4 * n for n in ns),
                    flops=case["iterations"] * sum(n * n * n + 3 * n * n for n in ns))
    n, m = case["n"], case["m"]
    if kind == "update":
        return dict(bytes=4 * m * (n + 1) + 8 * m + 16 * n * n, flops=2 * m * n + 3 * n * n)
    steps = case.get("iterations", 1)
    candidates = 2 * min(case.get("nn") or n, n) if case.get("nn") else n
    given = 0 if kind == "step" else 8 * n if case["coords"] else 4 * n * n
    return dict(bytes=given + 4 * n * n + 4 * n, flops=steps * (m * n * candidates + 3 * n * n))


# ---- the pheromone in 64 bits ---------------------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "update":
        a = _update_arrays(case, seed)
        n, rho = case["n"], RULES["as"][2]
        tau = (1.0 - rho) * a["tau"].astype(np.float64)
        edge = np.repeat(1.0 / a["lens"], n)
        np.add.at(tau, (a["tours"][:, :-1].ravel(), a["tours"][:, 1:].ravel()), edge)
        np.add.at(tau, (a["tours"][:, 1:].ravel(), a["tours"][:, :-1].ravel()), edge)
        return dict(tau=tau, choice=tau * a["heta"])
    plain = case["kind"] in ("solve", "step") and case["rule"] != "acs" and not case.get("nn") \
        and case.get("selection", "eq1") == "eq1"
    # about 20 seconds of small torch operations
    if not plain or case["m"] * case["n"] ** 2 * case.get("iterations", 1) > 2.5e10:
        return None
    return dict(tour=None, length=None, tau=_ant_system(case, seed))


_LOW = 0xFFFFFFFF


def _philox(step, ant, iteration, seed):
    """Words x0 and x1 of Philox4x32-10 at (step, ant, iteration, 0), as int64 tensors."""
    c = [step, ant, torch.full_like(step, iteration), torch.zeros_like(step)]
    k0, k1 = seed & _LOW, seed >> 32
    for r in range(10):
        p, q = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # the low 64 bits are what the shifts need
        c = [((q >> 32) & _LOW) ^ c[1] ^ k0, q & _LOW, ((p >> 32) & _LOW) ^ c[3] ^ k1, p & _LOW]
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    return c[0], c[1]


def _target(x0, x1, total):
    """floor((x1 2^32 + x0) total / 2^64) for total < 2^58."""
    th, tl = total >> 32, total & _LOW
    a, b, c = x1 * tl, x0 * th, x0 * tl
    mid = (a & _LOW) + (b & _LOW) + ((c >> 32) & _LOW)
    return x1 * th + ((a >> 32) & _LOW) + (b >> 32) + (mid >> 32)


def _power_of_two(e):
    return ((e.long() + 1023) << 52).view(torch.float64)


def _tours(choice, m, iteration, seed, lines):
    """The iteration's m closed tours by the integer roulette over float32 choice_info."""
    n, dev = choice.shape[0], choice.device
    ants = torch.arange(m, device=dev)
    x0, x1 = _philox(torch.arange(n, device=dev)[:, None].expand(n, m).contiguous(),
                     ants[None].expand(n, m).contiguous(), iteration, seed)
    cur = (x0[0] * n) >> 32
    seen = torch.zeros(m, n, dtype=torch.bool, device=dev)
    seen[ants, cur] = True
    tour = [cur]
    for s in range(1, n):
        w = choice[cur].masked_fill(seen, 0.0)
        e = torch.frexp(w.amax(1))[1]
        q = (w.double() * _power_of_two(46 - e)[:, None]).floor().long()
        sums = q.cumsum(1)
        t = _target(x0[s], x1[s], sums[:, -1])
        first_open = seen.to(torch.uint8).argmin(1)  # where every open weight is zero
        cur = torch.where(sums[:, -1] > 0, torch.searchsorted(sums, t[:, None], right=True)[:, 0],
                          first_open)
        seen[ants, cur] = True
        tour.append(cur)
    tour = torch.stack(tour + [tour[0]], 1)
    return tour, lines[tour[:, :-1], tour[:, 1:]].sum(1)


def _ant_system(case, seed):
    """float64 pheromone after the case's iterations (kernels keep it in float32, which decides the
    tours, so both are carried)."""
    n, m = case["n"], case["m"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    dist = torch.from_numpy(_instance(n, seed, case.get("clustered", False)).dist).to(dev).long()
    rho = float(np.float32(RULES[case["rule"]][2]))
    keep = float(np.float32(1.0) - np.float32(rho))
    off = ~torch.eye(n, dtype=torch.bool, device=dev)
    heta = torch.where(off, 1.0 / (dist * dist).clamp(min=1).double(), 0.0).float()
    d, left, at, nn_len = dist.cpu().numpy(), np.ones(n, bool), 0, 0
    for _ in range(n - 1):
        left[at] = False
        to = int(np.argmin(np.where(left, d[at], np.iinfo(np.int64).max)))
        nn_len, at = nn_len + int(d[at, to]), to
    nn_len += int(d[at, 0])
    mmas = case["rule"] == "mmas"
    root = P_BEST ** (1.0 / n)
    ratio = (1.0 - root) / ((n / 2.0 - 1.0) * root)

    def limits(best):
        top = 1.0 / (rho * best)
        return min(top * ratio, top), top

    tau64 = off.double() * (limits(nn_len)[1] if mmas else float(np.float32(m / nn_len)))
    tau32, best = tau64.float(), None
    for it in range(case.get("iterations", 1)):
        tour, lens = _tours(tau32 * heta, m, it, seed, dist)
        shortest, k = int(lens.min()), int(lens.argmin())
        best = shortest if best is None else min(best, shortest)
        if mmas:
            tour, lens = tour[k:k + 1], lens[k:k + 1]
        a, b = tour[:, :-1].reshape(-1), tour[:, 1:].reshape(-1)
        cells = torch.cat([a * n + b, b * n + a])
        each = (1.0 / lens.double())[:, None].expand(-1, n).reshape(-1).repeat(2)
        dep = torch.zeros(n * n, dtype=torch.float64, device=dev).index_add_(0, cells, each)
        tau64 = (1.0 - rho) * tau64 + dep.view(n, n)
        if mmas:
            add32 = dep.float().view(n, n)
            lo, hi = limits(best)
            lo32, hi32 = float(np.float32(lo)), float(np.float32(hi))
            tau32 = torch.where(off, (keep * tau32 + add32).clamp(lo32, hi32), 0.0)
            tau64 = torch.where(off, tau64.clamp(lo, hi), 0.0)
        else:
            # the deposit in fixed point, floor(dtau 2^shift) summed as whole numbers
            dtau = (1.0 / lens.double()).float()
            shift = 62 - (m - 1).bit_length() - (math.frexp(float(dtau.max()))[1] - 1)
            fixed = (dtau.double() * 2.0 ** shift).floor().long()[:, None].expand(-1, n).reshape(-1)
            total = torch.zeros(n * n, dtype=torch.int64, device=dev)
            total.index_add_(0, cells, fixed.repeat(2))
            tau32 = keep * tau32 + (total.float() * 2.0 ** -shift).view(n, n)
    return tau64
