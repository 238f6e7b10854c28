"""What a user of the library has it do, as measurable cases.

A case is one call pattern of the public package at one size:

  step     a kept solver is restarted from a vector and steps once (sfci_lanczos_load, sfci_lanczos_step):
           sigma = H w, the Lanczos scalars, the truncated next basis vector
  solve    the same from nothing: a solver is made for one vector, steps once, hands its vector over and is closed
  cycle    a kept solver runs one whole Lanczos cycle from a vector: its energies and the restart vector
  scan     one step of a batch of uneven systems advanced together
  sigma    the standalone sigma = H psi, every entry written out
  topk     the truncation of a long sparse vector to its largest entries
  rdm      the Rayleigh energy of a vector and its gradients with respect to the integrals (forward and backward)
  rank     determinants to indices and back

Integrals are drawn like those of the test systems (h: a diagonal spread of -2..1 with small off-diagonals; (pq|rs) from
Cholesky-like factors, 8-fold symmetric) or are the Hubbard ring's.  Vectors are drawn with the excitation levels and the spread
of magnitudes that truncated Lanczos vectors of these systems show after a few steps: a dense part around the lowest
determinant, where many determinants share a spin string, and a scattered part of higher pair excitations.
"""
import itertools
import math

import numpy as np
import torch

import paper_2312_01846_gb300 as sf

# share of the entries at each (alpha, beta) excitation level; the last two are the scattered part
LEVELS = {(1, 0): 0.005, (0, 1): 0.005, (2, 0): 0.03, (0, 2): 0.03, (1, 1): 0.14, (2, 1): 0.15, (1, 2): 0.15, (2, 2): 0.11,
          (3, 1): 0.05, (1, 3): 0.05, (3, 3): 0.10, (4, 4): 0.18}


def listed():
    return [
        # the whole space of 8 orbitals: the smallest solver call, where launches and host round trips count
        dict(name="step_8o_whole_space", kind="step", n=8, na=4, nb=4, factors=16, n_keep=4900, n_in=4900),
        # a cycle of the 12-site Hubbard ring with the paper's screen: short steps, nearly all integrals zero, dots over ten vectors
        dict(name="cycle_hubbard12_2e4", kind="cycle", n=12, na=6, nb=6, factors=0, n_keep=20000, n_in=20000, n_lanczos=10,
             eps_screen=5e-5),
        # float32 elements on the 28-orbital system at a small, odd vector length
        dict(name="step_28o_fp32_20011", kind="step", n=28, na=7, nb=7, factors=200, n_keep=20011, n_in=20011, fp32=True),
        # the everyday step: 28 orbitals, 5e4 determinants
        dict(name="step_28o_5e4", kind="step", n=28, na=7, nb=7, factors=200, n_keep=50000, n_in=50000),
        # the largest vector: a solver of 3e5 determinants made, stepped and closed
        dict(name="solve_28o_3e5", kind="solve", n=28, na=7, nb=7, factors=200, n_keep=300000, n_in=300000),
        # a scan along a parameter: 32 systems of 16 to 24 orbitals, 5 to 8 electrons per spin, small and uneven vectors
        dict(name="scan_32_systems", kind="scan", count=32, n_max=24, cap_lo=500, cap_hi=10000),
        # the standalone product on a short vector and on a long one (20 orbitals)
        dict(name="sigma_20o_601", kind="sigma", n=20, na=5, nb=5, factors=64, n_in=601),
        dict(name="sigma_20o_6000", kind="sigma", n=20, na=5, nb=5, factors=64, n_in=6000),
        # the standalone truncation of a long vector
        dict(name="topk_3e6_to_2e5", kind="topk", n_in=3000001, k=200000),
        # gradients of the energy: a short vector, and the 3e5 determinants of a converged one
        dict(name="rdm_20o_1201", kind="rdm", n=20, na=5, nb=5, factors=64, n_in=1201),
        dict(name="rdm_20o_3e5", kind="rdm", n=20, na=5, nb=5, factors=64, n_in=300000),
        # indexing of a million determinants both ways
        dict(name="rank_28o_1e6", kind="rank", n=28, na=7, nb=7, n_in=1000003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "cycle", "sigma", "topk", "rdm", "rank"])
    n = rng.randint(14, 28)
    na = rng.randint(3, 7)
    nb = rng.choice([na, na, max(2, na - 1), min(7, na + 1)])
    base = dict(kind=kind, n=n, na=na, nb=nb, factors=rng.choice([16, 64, 200]))
    space = math.comb(n, na) * math.comb(n, nb) // 8
    if kind in ("step", "cycle"):
        keep = min(_log_int(rng, 300, 60000 if kind == "step" else 12000), space)
        base.update(n_keep=keep, n_in=max(1, int(keep * rng.choice([1.0, 1.0, 0.37]))))
        if rng.random() < 0.25:
            base["fp32"] = True
        if rng.random() < 0.25:
            base["eps_screen"] = 5e-5
        if kind == "cycle":
            base["n_lanczos"] = rng.randint(3, 10)
        return base
    if kind == "sigma":
        n = rng.randint(12, 20)
        na = rng.randint(3, 5)
        return dict(kind=kind, n=n, na=na, nb=na, factors=16,
                    n_in=min(_log_int(rng, 20, 5000), math.comb(n, na) ** 2 // 8))
    if kind == "rdm":
        n = rng.randint(12, 20)
        na = rng.randint(3, 5)
        return dict(kind=kind, n=n, na=na, nb=na, factors=16,
                    n_in=min(_log_int(rng, 100, 200000), math.comb(n, na) ** 2 // 8))
    if kind == "topk":
        n_in = _log_int(rng, 1000, 3000000)
        return dict(kind=kind, n_in=n_in, k=max(1, int(n_in * math.exp(rng.uniform(math.log(0.003), math.log(0.9))))))
    return dict(kind=kind, n=n, na=na, nb=nb, n_in=_log_int(rng, 1000, 2000000))


# ---------------------------------------------------------------- inputs

def _integrals(case, seed):
    n = case["n"]
    rng = np.random.default_rng(seed)
    if not case["factors"]:  # the Hubbard ring (its strength from the seed, around U = 4 t)
        h = np.zeros((n, n))
        for i in range(n):
            h[i, (i + 1) % n] = h[(i + 1) % n, i] = -1.0
        g = np.zeros((n, n, n, n))
        for p in range(n):
            g[p, p, p, p] = 3.5 + rng.random()
        return h, g
    return _molecular(rng, n, case["factors"], cluster=n >= 26)


def _molecular(rng, n, factors, cluster=False):
    h = np.triu(rng.normal(0.0, 0.1, (n, n)), 1)
    h = h + h.T
    if cluster:
        diag = np.concatenate([np.sort(rng.uniform(-2.0, -1.9, n // 2)), np.sort(rng.uniform(0.9, 1.0, n - n // 2))])
    else:
        diag = np.linspace(-2.0, 1.0, n)
    h[np.diag_indices(n)] = diag
    p, q = np.tril_indices(n)
    b = rng.normal(0.0, 0.3, (factors, p.size))
    m = b.T @ b  # (pair | pair), made exactly symmetric
    m = np.tril(m) + np.tril(m, -1).T
    pair = np.zeros((n, n), dtype=np.int64)
    pair[p, q] = pair[q, p] = np.arange(p.size)
    g = m[pair[:, :, None, None], pair[None, None, :, :]]
    return h, np.ascontiguousarray(g)


def _excited(gen, n, m, level):
    """One spin string per entry of `level`: that many electrons of the lowest string moved to random empty orbitals."""
    size = level.numel()
    out = torch.full((size,), (1 << m) - 1, dtype=torch.int64, device="cuda")
    kmax = min(int(level.max()), m, n - m) if size else 0
    if kmax == 0:
        return out
    holes = torch.rand((size, m), generator=gen, device="cuda").topk(kmax, dim=1).indices
    parts = torch.rand((size, n - m), generator=gen, device="cuda").topk(kmax, dim=1).indices + m
    for k in range(kmax):
        move = (torch.ones_like(out) << holes[:, k]) | (torch.ones_like(out) << parts[:, k])
        out = torch.where(level > k, out ^ move, out)
    return out


def _string_index(s, n, m):
    """Colexicographic index of each spin string."""
    table = torch.tensor([[math.comb(b, k) for k in range(m + 1)] for b in range(n)], dtype=torch.int64, device=s.device)
    out = torch.zeros_like(s)
    seen = torch.zeros_like(s)
    for b in range(n):
        bit = (s >> b) & 1
        seen += bit
        out += bit * table[b][seen]
    return out


def _determinants(case, seed, count):
    """`count` distinct determinants (alpha, beta, level) sorted by index, the lowest one among them."""
    n, na, nb = case["n"], case["na"], case["nb"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    pairs = torch.tensor(list(LEVELS), device="cuda")
    share = torch.tensor(list(LEVELS.values()), device="cuda")
    cb = math.comb(n, nb)
    alpha = torch.tensor([(1 << na) - 1], device="cuda")
    beta = torch.tensor([(1 << nb) - 1], device="cuda")
    index = torch.zeros(1, dtype=torch.int64, device="cuda")
    uniform = 0.0  # share of determinants drawn from the whole space, raised where the levels run dry
    while index.numel() < count:
        size = 2 * (count - index.numel()) + 64
        lev = pairs[torch.multinomial(share, size, replacement=True, generator=gen)]
        wide = torch.rand(size, generator=gen, device="cuda") < uniform
        a = _excited(gen, n, na, torch.where(wide, n, lev[:, 0]))
        b = _excited(gen, n, nb, torch.where(wide, n, lev[:, 1]))
        if uniform:
            ra = torch.rand((size, n), generator=gen, device="cuda").topk(na, dim=1).indices
            rb = torch.rand((size, n), generator=gen, device="cuda").topk(nb, dim=1).indices
            a = torch.where(wide, (torch.ones_like(ra) << ra).sum(1), a)
            b = torch.where(wide, (torch.ones_like(rb) << rb).sum(1), b)
        k = _string_index(a, n, na) * cb + _string_index(b, n, nb)
        new = torch.unique(torch.cat([index, k]))
        fresh = new[~torch.isin(new, index)]
        if fresh.numel() > count - index.numel():
            pick = torch.randperm(fresh.numel(), generator=gen, device="cuda")[: count - index.numel()]
            fresh = fresh[pick]
        where = torch.argsort(k)
        at = where[torch.searchsorted(k[where], fresh)]
        alpha, beta, index = torch.cat([alpha, a[at]]), torch.cat([beta, b[at]]), torch.cat([index, fresh])
        uniform = min(1.0, uniform + 0.2)
    order = torch.argsort(index)
    return alpha[order], beta[order], index[order]


def _vector(case, seed):
    """A normalised sparse vector of n_in entries: (alpha, beta, index, coefficient)."""
    n, na, nb, count = case["n"], case["na"], case["nb"], case["n_in"]
    dim = math.comb(n, na) * math.comb(n, nb)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 77)
    if count >= dim:
        index = torch.arange(dim, device="cuda")
        strings = [torch.tensor(sorted(sum(1 << o for o in c) for c in itertools.combinations(range(n), m)), device="cuda")
                   for m in (na, nb)]
        cb = math.comb(n, nb)
        alpha, beta = strings[0][index // cb], strings[1][index % cb]
    else:
        # (the number of entries of a standalone sigma depends on the determinants alone: they belong to the case)
        alpha, beta, index = _determinants(case, 1 if case.get("kind") == "sigma" else seed, count)
    one = torch.ones_like(alpha)
    level = torch.zeros_like(alpha)
    for b in range(n):
        level += ((alpha >> b) & one) * (1 if b >= na else 0) + ((beta >> b) & one) * (1 if b >= nb else 0)
    size = index.numel()
    mag = torch.exp(-0.7 * level.clamp(max=5).double()
                    + 0.6 * torch.randn(size, generator=gen, device="cuda", dtype=torch.float64))
    sign = torch.randint(0, 2, (size,), generator=gen, device="cuda") * 2 - 1
    coef = mag * sign
    return alpha, beta, index, coef / coef.norm()


def _system(case, seed):
    h, g = _integrals(case, seed)
    return sf.System(case["n"], case["na"], case["nb"], h, g, 0.0, sf.SFCI_FP32_ELEMENTS if case.get("fp32") else 0)


def _scan_instances(case, seed):
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(3)  # the systems' sizes belong to the case, their integrals and vectors to the seed
    n_max, count = case["n_max"], case["count"]
    h0, g0 = _molecular(rng, n_max, 16)
    h1, g1 = _molecular(rng, n_max, 16)
    out = []
    for i in range(count):
        lam = i / max(count - 1, 1)
        n, ne = int(sizes.integers(16, n_max + 1)), int(sizes.integers(5, 9))
        cap = int(round(math.exp(sizes.uniform(math.log(case["cap_lo"]), math.log(case["cap_hi"])))))
        h = ((1 - lam) * h0 + lam * h1)[:n, :n]
        g = ((1 - lam) * g0 + lam * g1)[:n, :n, :n, :n]
        _, _, index, coef = _vector(dict(n=n, na=ne, nb=ne, n_in=cap), seed + i)
        out.append((sf.System(n, ne, ne, np.ascontiguousarray(h), np.ascontiguousarray(g)), index, coef, cap))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "scan":
        return dict(case=case, scan=sf.Scan(_scan_instances(case, seed), n_lanczos=10))
    if kind == "topk":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        size = case["n_in"]
        rank = torch.randint(0, 1 << 40, (size,), generator=gen, device="cuda") // 4 * 4 + torch.arange(size, device="cuda") % 4
        rank = torch.unique(rank)
        while rank.numel() < size:
            more = torch.randint(0, 1 << 40, (2 * (size - rank.numel()),), generator=gen, device="cuda")
            rank = torch.unique(torch.cat([rank, more]))[:size]
        coef = torch.randn(size, generator=gen, device="cuda", dtype=torch.float64)
        coef = coef * torch.exp(2.0 * torch.randn(size, generator=gen, device="cuda", dtype=torch.float64) - 8.0)
        perm = torch.randperm(size, generator=gen, device="cuda")  # unsorted, as a merge leaves it
        return dict(case=case, rank=rank[perm], coef=coef)
    if kind == "rank":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        strings = [(torch.ones((case["n_in"], m), dtype=torch.int64, device="cuda")
                    << torch.rand((case["n_in"], case["n"]), generator=gen, device="cuda").topk(m, dim=1).indices).sum(1)
                   for m in (case["na"], case["nb"])]
        n = case["n"]
        sys_ = sf.System(n, case["na"], case["nb"], np.zeros((n, n)), np.zeros((n, n, n, n)))
        return dict(case=case, sys=sys_, alpha=strings[0], beta=strings[1])
    state = dict(case=case, sys=_system(case, seed))
    _, _, state["rank"], state["coef"] = _vector(case, seed)
    if kind in ("step", "cycle"):
        state["solver"] = sf.Lanczos(state["sys"], state["rank"], state["coef"], case["n_keep"],
                                     n_lanczos=case.get("n_lanczos", 10), eps_screen=case.get("eps_screen", 0.0))
    if kind == "rdm":
        h, g = _integrals(case, seed)
        state["h"], state["g"] = torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda()
    return state


# ---------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "scan":
        scan = state["scan"]
        infos = scan.step()
        vecs = [scan.vector(i) for i in range(scan.count)]
        return dict(rank=torch.cat([r for r, _ in vecs]), coef=torch.cat([c for _, c in vecs]),
                    a=np.array([x["a"] for x in infos]), energy=np.array([x["lambda_min"] for x in infos]))
    if kind == "topk":
        rank, coef = sf.sfci_truncate_topk(state["rank"], state["coef"], case["k"])
        return dict(rank=rank, coef=coef)
    if kind == "rank":
        rank = sf.sfci_rank(state["sys"], state["alpha"], state["beta"])
        alpha, beta = sf.sfci_unrank(state["sys"], rank)
        return dict(rank=rank, alpha=alpha, beta=beta)
    if kind == "sigma":
        rank, coef = sf.sfci_sigma(state["sys"], state["rank"], state["coef"])
        return dict(rank=rank, coef=coef)
    if kind == "rdm":
        h = state["h"].clone().requires_grad_()
        g = state["g"].clone().requires_grad_()
        energy = sf.RayleighEnergy.apply(h, g, state["sys"], state["rank"], state["coef"])
        dh, dg = torch.autograd.grad(energy, (h, g))
        return dict(energy=energy, dh=dh, dg=dg)
    if kind == "solve":
        solver = sf.Lanczos(state["sys"], state["rank"], state["coef"], case["n_keep"])
        info = solver.step()
        rank, coef = solver.vector()
        solver.close()
        return dict(rank=rank, coef=coef, a=np.array(info["a"]), u_norm=np.array(info["u_norm"]))
    solver = state["solver"]
    solver.load(state["rank"], state["coef"])
    if kind == "step":
        info = solver.step()
        rank, coef = solver.vector()
        return dict(rank=rank, coef=coef, a=np.array(info["a"]), u_norm=np.array(info["u_norm"]))
    infos = [solver.step() for _ in range(case["n_lanczos"])]
    rank, coef = solver.vector()
    return dict(rank=rank, coef=coef, energy=np.array(infos[-1]["lambda_min"]), a=np.array([x["a"] for x in infos]),
                b=np.array([x["b"] for x in infos]))


# ---------------------------------------------------------------- what a pass cannot do without

def _connected(n, na, nb):
    sa, sb = na * (n - na), nb * (n - nb)
    return 1 + sa + sb + sa * sb + math.comb(na, 2) * math.comb(n - na, 2) + math.comb(nb, 2) * math.comb(n - nb, 2)


def work(case):
    kind = case["kind"]
    if kind == "topk":
        return dict(bytes=16 * (case["n_in"] + min(case["k"], case["n_in"])), flops=3 * min(case["k"], case["n_in"]))
    if kind == "rank":
        return dict(bytes=5 * 8 * case["n_in"], flops=2 * (case["na"] + case["nb"]) * case["n_in"])
    if kind == "scan":  # the mean size of the drawn instances
        n_in = case["count"] * (case["cap_hi"] - case["cap_lo"]) / math.log(case["cap_hi"] / case["cap_lo"])
        return dict(bytes=int(32 * n_in), flops=int(2 * n_in * _connected((16 + case["n_max"]) // 2, 6, 6)))
    n, n_in = case["n"], case["n_in"]
    elements = n_in * _connected(n, case["na"], case["nb"])
    tables = 8 * (n ** 4 + n ** 2)
    if kind == "sigma":  # an entry is made of a few elements
        return dict(bytes=tables + 16 * n_in + 16 * min(elements // 2, math.comb(n, case["na"]) * math.comb(n, case["nb"])),
                    flops=2 * elements)
    if kind == "rdm":
        return dict(bytes=2 * tables + 16 * n_in, flops=2 * elements)
    steps = case.get("n_lanczos", 1) if kind == "cycle" else 1
    if not case["factors"]:  # the ring: hops to the neighbouring sites only
        elements = n_in * (1 + 2 * (case["na"] + case["nb"]))
    return dict(bytes=tables + 16 * n_in + 16 * steps * case["n_keep"], flops=2 * steps * elements)


# ---------------------------------------------------------------- the same in plain numpy

def _sign_below(s, p):
    """(-1) ** (occupied orbitals of s below p), per string."""
    x = s & ((1 << p) - 1)
    sign = np.ones(s.shape)
    while np.any(x):
        sign = np.where(x & 1, -sign, sign)
        x = x >> 1
    return sign


def _replace(s, p, q):
    """a+_p a_q on spin strings: (which survive, the new strings, their signs)."""
    ok = ((s >> q) & 1) == 1
    t = s[ok] ^ (1 << q)
    sign = _sign_below(t, q)
    free = ((t >> p) & 1) == 0
    ok = np.nonzero(ok)[0][free]
    t, sign = t[free], sign[free]
    return ok, t | (1 << p), sign * _sign_below(t, p)


def _np_index(s, n, m):
    return _string_index(torch.from_numpy(np.ascontiguousarray(s)), n, m).numpy()


def _replaced(alpha, beta, n, na, nb):
    """Every E_pq |D> of a list of determinants: (pq, source, index, alpha, beta, sign), E_pq = sum of a+_p a_q over both spins."""
    cb = math.comb(n, nb)
    ia, ib = _np_index(alpha, n, na), _np_index(beta, n, nb)
    rows = []
    for p in range(n):
        for q in range(n):
            ok, t, s = _replace(alpha, p, q)
            rows.append((np.full(ok.size, p * n + q), ok, _np_index(t, n, na) * cb + ib[ok], t, beta[ok], s))
            ok, t, s = _replace(beta, p, q)
            rows.append((np.full(ok.size, p * n + q), ok, ia[ok] * cb + _np_index(t, n, nb), alpha[ok], t, s))
    return [np.concatenate(x) for x in zip(*rows)]


def _exact_sigma(case, h, g, alpha, beta, coef):
    """H psi = sum h'_pq E_pq psi + 1/2 sum (pq|rs) E_pq E_rs psi, through the determinants that the E_rs reach."""
    n, na, nb = case["n"], case["na"], case["nb"]
    pq, src, index, a1, b1, s = _replaced(alpha, beta, n, na, nb)
    mid, first, inv = np.unique(index, return_index=True, return_inverse=True)
    d = np.zeros((mid.size, n * n))  # d[K, rs] = <K|E_rs|psi>
    np.add.at(d, (inv, pq), s * coef[src])
    hp = h - 0.5 * np.einsum("prrq->pq", g)
    v = 0.5 * d @ g.reshape(n * n, n * n).T
    pq2, src2, index2, _, _, s2 = _replaced(a1[first], b1[first], n, na, nb)
    top, inv2 = np.unique(index2, return_inverse=True)
    out = np.bincount(inv2, s2 * v[src2, pq2], top.size)
    out[np.searchsorted(top, mid)] += d @ hp.reshape(n * n)
    return top, out


def exact(case, seed):
    kind = case["kind"]
    if kind == "rank":
        s = prepare(case, seed)
        cb = math.comb(case["n"], case["nb"])
        rank = _string_index(s["alpha"], case["n"], case["na"]) * cb + _string_index(s["beta"], case["n"], case["nb"])
        return dict(rank=rank.cpu(), alpha=s["alpha"].cpu(), beta=s["beta"].cpu())
    if kind == "topk":
        s = prepare(case, seed)
        rank, coef = s["rank"].cpu().numpy(), s["coef"].cpu().numpy()
        keep = np.lexsort((rank, -np.abs(coef)))[: case["k"]]
        keep = np.sort(keep[coef[keep] != 0.0])
        keep = keep[np.argsort(rank[keep])]
        return dict(rank=rank[keep], coef=coef[keep] / np.sqrt(np.sum(coef[keep].astype(np.longdouble) ** 2)).astype(np.float64))
    if kind not in ("sigma", "step", "rdm") or case.get("eps_screen") or case.get("fp32"):
        return None
    if case["n_in"] * case["n"] ** 2 > 600000 or not case["factors"]:
        return None
    n, na, nb = case["n"], case["na"], case["nb"]
    h, g = _integrals(case, seed)
    alpha, beta, index, coef = (x.cpu().numpy() for x in _vector(case, seed))
    if kind == "sigma":
        rank, val = _exact_sigma(case, h, g, alpha, beta, coef)
        return dict(rank=rank, coef=val)
    if kind == "rdm":
        pq, src, key, _, _, s = _replaced(alpha, beta, n, na, nb)
        mid, inv = np.unique(key, return_inverse=True)
        d = np.zeros((mid.size, n * n))
        np.add.at(d, (inv, pq), s * coef[src])
        norm = float(coef @ coef)
        at = np.searchsorted(mid, index)  # psi's own entries among the determinants reached
        gamma = (coef @ d[at]).reshape(n, n)  # <psi|E_pq|psi>
        two = (d.T @ d).reshape(n, n, n, n).transpose(1, 0, 2, 3).copy()  # <E_qp psi|E_rs psi>
        for q in range(n):
            two[:, q, q, :] -= gamma
        energy = (np.sum(h * gamma) + 0.5 * np.sum(g * two)) / norm
        return dict(energy=np.array(energy), dh=gamma / norm, dg=0.5 * two / norm)
    rank, val = _exact_sigma(case, h, g, alpha, beta, coef)
    on = np.searchsorted(rank, index)
    a = float(coef @ val[on])
    u = val.copy()
    u[on] -= a * coef
    keep = np.lexsort((rank, -np.abs(u)))[: case["n_keep"]]
    keep = np.sort(keep[u[keep] != 0.0])
    return dict(rank=rank[keep], coef=u[keep] / np.linalg.norm(u[keep]), a=np.array(a), u_norm=np.array(np.linalg.norm(u)))
