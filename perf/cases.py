"""Workloads of the EN-PT2 / CIPSI library, for timing and for comparing results.

A case names an entry point and its sizes; ``prepare`` makes its Hamiltonian
and wave function from a seed, ``run`` makes one call through the package's
public functions, ``work`` gives the bytes and FP64 operations the call cannot
do without, and ``exact`` evaluates the same quantities in plain FP64 torch
(every substitution of every internal determinant, grouped by determinant)
where that takes seconds.

Hamiltonians follow the recipe of the package's synthetic inputs (decaying
Cholesky vectors, h_pp = -2 + 0.15 p).  Wave functions look like CIPSI spaces:
the determinants of largest first-order amplitude among the singles and
doubles of the reference and the products of two of them, with coefficients
near those amplitudes (a few per cent of noise keeps spin partners from tying).
"""
import math

import numpy as np
import torch

import paper_1902_08154_gb300 as qp

DECAY = 0.9048374180359595  # exp(-0.1)


def listed():
    return [
        # the first iterations of a CIPSI run: a few dozen determinants in host
        # arrays, per-generator sums wanted (launches and copies are the cost)
        dict(name="first_iterations", kind="sweep", norb=16, na=4, nb=4, ndet=50, k=100, mixed=False, host=True),
        # an early iteration of an open shell, on the device
        dict(name="early_open_shell", kind="sweep", norb=24, na=6, nb=5, ndet=150, k=300, mixed=False, host=False),
        # odd sizes in the middle of a run
        dict(name="middle_ragged", kind="sweep", norb=47, na=9, nb=8, ndet=1201, k=2401, mixed=False, host=False),
        # the full-size sweep of a 64-orbital active space (the benchmark's shape)
        dict(name="full_64", kind="sweep", norb=64, na=10, nb=10, ndet=10000, k=20000, mixed=False, host=False),
        # the mixed-precision sweep, chosen where 1e-6 Eh is enough
        dict(name="mixed_56", kind="sweep", norb=56, na=9, nb=9, ndet=3000, k=6000, mixed=True, host=False),
        # two words per spin: the largest orbital count
        dict(name="two_words_128", kind="sweep", norb=128, na=14, nb=14, ndet=1000, k=1000, mixed=False, host=False),
        # one draw of the hybrid stochastic E_PT2: a few generators of a large space
        dict(name="generators_64", kind="gens", norb=64, na=10, nb=10, ndet=10000, ngen=240),
        # the gradient with respect to the integrals (orbital optimisation)
        dict(name="gradient_48", kind="grad", norb=48, na=8, nb=8, ndet=2000),
        # two states at once, with the multi-state selection
        dict(name="two_states_64", kind="states", norb=64, na=10, nb=10, ndet=2000, k=4000, nst=2),
        # the variational step that follows every sweep
        dict(name="davidson_64", kind="davidson", norb=64, na=10, nb=10, ndet=10000),
        # many uneven instances in one graph (geometry scans)
        dict(name="batch_uneven", kind="batch", n=10, size=400),
        # the entry point for callers that may not allocate
        dict(name="noalloc_32", kind="noalloc", norb=32, na=6, nb=6, ndet=300, k=300),
    ]


def substitutions(norb, na, nb):
    va, vb = norb - na, norb - nb
    return (na * va + nb * vb + math.comb(na, 2) * math.comb(va, 2) + math.comb(nb, 2) * math.comb(vb, 2)
            + na * nb * va * vb)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "sweep", "gens", "grad", "states", "davidson", "batch", "noalloc"])
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(2, 12), size=_log_int(rng, 60, 500))
    limit = {"sweep": 2.0e9, "gens": 2.0e9, "grad": 1.5e8, "states": 4.0e8, "noalloc": 1.0e8, "davidson": 4.0e9}[kind]
    while True:
        norb = rng.randint(14, 40) if kind == "noalloc" else rng.randint(14, 64) if rng.random() < 0.8 else rng.randint(65, 128)
        na = rng.randint(3, min(14, norb // 3))
        nb = max(2, na - rng.choice([0, 0, 1, 2]))
        ndet = _log_int(rng, 40, 300 if kind == "noalloc" else 10000)
        case = dict(kind=kind, norb=norb, na=na, nb=nb, ndet=ndet)
        nsd = substitutions(norb, na, nb)
        if kind == "gens":
            case["ngen"] = min(ndet, _log_int(rng, 8, 400))
            cost = case["ngen"] * nsd
        else:
            cost = ndet * nsd
        if norb > 64:
            cost *= 3
        if cost > limit or nsd < 4 * ndet:
            continue
        if kind in ("sweep", "states", "noalloc"):
            case["k"] = rng.choice([0, ndet, 2 * ndet - 1]) if kind == "sweep" else ndet
        if kind == "sweep":
            case["mixed"] = rng.random() < 0.25
            case["host"] = rng.random() < 0.3
        if kind == "states":
            case["nst"] = rng.choice([2, 3] if norb <= 64 else [2])
        return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _hamiltonian(norb, rank, rng):
    """h [norb, norb], V [pairs, pairs] with V[pq, rs] = (pq|rs), packed eri."""
    dev = "cuda"
    up = torch.from_numpy(rng.normal(0.0, 0.05, size=(norb, norb))).to(dev).triu(1)
    h = up + up.T + torch.diag(-2.0 + 0.15 * torch.arange(norb, dtype=torch.float64, device=dev))
    p, q = torch.tril_indices(norb, norb, device=dev)
    scale = 0.3 * torch.pow(torch.tensor(DECAY, dtype=torch.float64, device=dev), (p + q).double())
    B = torch.from_numpy(rng.standard_normal((rank, p.numel()))).to(dev) * scale
    V = B.T @ B
    V = torch.tril(V) + torch.tril(V, -1).T
    r, c = torch.tril_indices(p.numel(), p.numel(), device=dev)
    return h.contiguous(), V, V[r, c].contiguous()


def _pair(p, q):
    hi, lo = torch.maximum(p, q), torch.minimum(p, q)
    return hi * (hi + 1) // 2 + lo


def _bits(norb, nint, spin, orb):
    """One spin orbital as words [..., 2 * nint]."""
    words = torch.zeros(orb.shape + (2 * nint,), dtype=torch.int64, device=orb.device)
    one = torch.ones_like(orb)
    return words.scatter_(-1, (spin * nint + orb // 64).unsqueeze(-1), torch.bitwise_left_shift(one, orb % 64).unsqueeze(-1))


def _mixed_key(words):
    """64-bit hash of determinant words (wrapping arithmetic)."""
    k = torch.zeros(words.shape[:-1], dtype=torch.int64, device=words.device)
    for w in range(words.shape[-1]):
        k = (k ^ words[..., w]) * -7046029254386353131
        k = k ^ ((k >> 29) & 0x7FFFFFFFF)
        k = k * -4658895280553007687
        k = k ^ ((k >> 32) & 0xFFFFFFFF)
    return k


def _space(norb, na, nb, ndet, h, V, rng):
    """Determinants [ndet, 2, nint], coefficients and E0 (see the file header)."""
    dev, nint = h.device, (norb - 1) // 64 + 1
    orb = torch.arange(norb, device=dev)
    diag = _pair(orb, orb)
    J = V[diag][:, diag]
    pq = _pair(orb[:, None], orb[None, :])
    K = V[pq, pq]
    nocc = (na, nb)
    occ = [(orb < n).double() for n in nocc]
    F = []
    for s in range(2):
        f = h.clone()
        for t in range(2):
            for j in range(nocc[t]):
                f = f + V[pq, diag[j]]
                if t == s:
                    f = f - V[pq[:, j][:, None], pq[:, j][None, :]]
        F.append(f)
    e_hf = sum(float((occ[s] * (torch.diag(h) + torch.diag(F[s]))).sum()) for s in range(2)) / 2
    amps, holes, parts = [], [], []

    def add(t, hs, ps):
        amps.append(t.reshape(-1))
        holes.append(torch.stack([x.expand(t.shape).reshape(-1) for x in hs], -1))
        parts.append(torch.stack([x.expand(t.shape).reshape(-1) for x in ps], -1))

    none = torch.full((1,), -1, device=dev)
    for s in range(2):  # singles and same-spin doubles; codes are s * norb + orbital
        n, e = nocc[s], torch.diag(F[s])
        i, a = orb[:n], orb[n:]
        ii, aa = i[:, None], a[None, :]
        add(F[s][ii, aa] / (e[ii] - e[aa]), (s * norb + ii, none), (s * norb + aa, none))
        if n > 1:
            i2, j2 = torch.triu_indices(n, n, 1, device=dev)
            a2, b2 = torch.triu_indices(norb - n, norb - n, 1, device=dev) + n
            i2, j2, a2, b2 = i2[:, None], j2[:, None], a2[None, :], b2[None, :]
            v = V[_pair(i2, a2), _pair(j2, b2)] - V[_pair(i2, b2), _pair(j2, a2)]
            add(v / (e[i2] + e[j2] - e[a2] - e[b2]), (s * norb + i2, s * norb + j2), (s * norb + a2, s * norb + b2))
    ea, eb = torch.diag(F[0]), torch.diag(F[1])
    i = orb[:na][:, None, None, None]
    j = orb[:nb][None, :, None, None]
    a = orb[na:][None, None, :, None]
    b = orb[nb:][None, None, None, :]
    add(V[_pair(i, a), _pair(j, b)] / (ea[i] + eb[j] - ea[a] - eb[b]), (i, norb + j), (a, norb + b))
    amp, hol, par = torch.cat(amps), torch.cat(holes), torch.cat(parts)
    keep = torch.topk(amp.abs(), min(amp.numel(), ndet + 1200)).indices
    amp, hol, par = amp[keep], hol[keep], par[keep]

    def mask(codes):
        w = torch.zeros((len(codes), 2 * nint), dtype=torch.int64, device=dev)
        for c in codes.unbind(-1):
            ok = c >= 0
            c = torch.where(ok, c, 0)
            w = w | torch.where(ok[:, None], _bits(norb, nint, c // norb, c % norb), 0)
        return w

    mh, mp = mask(hol), mask(par)
    m = min(len(amp), 1200)
    u, v = torch.triu_indices(m, m, 1, device=dev)
    clash = ((mh[u] & mh[v]) | (mp[u] & mp[v])).ne(0).any(-1)
    u, v = u[~clash], v[~clash]
    amp = torch.cat([torch.ones(1, dtype=torch.float64, device=dev), amp, amp[u] * amp[v]])
    flip = torch.cat([torch.zeros((1, 2 * nint), dtype=torch.int64, device=dev), mh | mp, (mh | mp)[u] ^ (mh | mp)[v]])
    order = torch.argsort(amp.abs(), descending=True, stable=True)[: 4 * ndet + 64]
    amp, flip = amp[order], flip[order]
    _, inv = torch.unique(_mixed_key(flip), return_inverse=True)
    first = torch.full((int(inv.max()) + 1,), len(inv), device=dev)
    first = first.scatter_reduce(0, inv, torch.arange(len(inv), device=dev), "amin")
    first = torch.sort(first).values[:ndet]
    if len(first) < ndet:
        raise ValueError("space too small for the requested number of determinants")
    hf = sum(_bits(norb, nint, torch.full((n,), s, device=dev), orb[:n]).sum(0) for s, n in enumerate(nocc))
    dets = (hf[None, :] ^ flip[first]).reshape(ndet, 2, nint).contiguous()
    c = amp[first] * (1.0 + 0.05 * torch.from_numpy(rng.standard_normal(ndet)).to(dev))
    c = c / c.norm()
    return dets, c.contiguous(), e_hf - 1.0 - 0.1 * norb / 16


def _instance(case, seed, nst=1):
    rng = np.random.default_rng(seed)
    norb = case["norb"]
    h, V, eri = _hamiltonian(norb, norb + norb // 2, rng)
    dets, c, e0 = _space(norb, case["na"], case["nb"], case["ndet"], h, V, rng)
    coefs = [c]
    for _ in range(nst - 1):  # further states: weight moved to other determinants
        d = c[torch.from_numpy(rng.permutation(len(c))).to(c.device)] + 0.2 * c
        coefs.append(d / d.norm())
    return h, V, eri, dets, (c if nst == 1 else torch.stack(coefs)), e0


def _batch_sizes(case):
    rng = np.random.default_rng(1000 * case["n"] + case["size"])
    out = []
    for i in range(case["n"]):
        norb = int(rng.choice([24, 32, 48, 64, 72]))
        ne = int(rng.integers(5, 10 if norb > 24 else 8))
        ndet = max(24, int(case["size"] * math.exp(rng.uniform(-1.5, 0.5))))
        out.append(dict(norb=norb, na=ne, nb=ne, ndet=ndet, k=ndet))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        insts = []
        for i, c in enumerate(_batch_sizes(case)):
            h, _, eri, dets, coefs, e0 = _instance(c, seed * 100 + i)
            pt2 = qp.PT2(c["norb"], c["na"], c["nb"], h, eri)
            insts.append(dict(pt2=pt2, dets=dets, coefs=coefs, e0=e0, k=c["k"]))
        return dict(kind=kind, batch=qp.Batch(insts))
    h, _, eri, dets, coefs, e0 = _instance(case, seed, case.get("nst", 1))
    st = dict(kind=kind, case=case, dets=dets, coefs=coefs, e0=e0)
    if kind == "noalloc":
        k = case["k"]
        st.update(h=h, eri=eri, sel=torch.zeros_like(dets[:1]).repeat(k, 1, 1), se=torch.zeros(k, dtype=torch.float64, device="cuda"))
        return st
    st["pt2"] = qp.PT2(case["norb"], case["na"], case["nb"], h, eri, precision=qp.QP_MIXED if case.get("mixed") else qp.QP_FP64)
    if kind == "sweep" and case["host"]:
        st.update(dets=dets.cpu().numpy().view(np.uint64), coefs=coefs.cpu().numpy())
    if kind == "gens":  # ranks drawn by weight, as the stochastic estimator does
        w = (coefs * coefs).cpu().numpy()
        st["ranks"] = np.random.default_rng(seed + 5).choice(len(w), size=case["ngen"], replace=False, p=np.sort(w)[::-1] / w.sum()).astype(np.int32)
    if kind == "states":
        st["e0"] = e0 - 0.2 * np.arange(case["nst"])
    if kind == "grad":
        st.update(dh=torch.zeros_like(h), deri=torch.zeros_like(eri))
    return st


def _signed(x):
    return x - (1 << 64) if x >= (1 << 63) else x


TOTALS = ("e_pt2", "sum_e_over_d", "min_abs_den", "z", "e_rpt2", "n_perturbers", "n_connections", "n_selected", "n_tiny")


def _totals(d):
    out = {f: d[f] for f in TOTALS}
    out["digest"] = [_signed(x) for x in d["digest"]]
    return out


def _array(x):
    return x.view(np.int64) if isinstance(x, np.ndarray) and x.dtype == np.uint64 else x


def run(state):
    kind = state["kind"]
    if kind == "batch":
        out, _ = state["batch"].run()
        return dict(
            energies=np.array([[d[f] for f in TOTALS[:5]] for d in out]),
            counts=np.array([[d[f] for f in TOTALS[5:]] + [_signed(x) for x in d["digest"]] for d in out]),
            sel_dets=[d["sel_dets"] for d in out], sel_e=[d["sel_e"] for d in out])
    case, dets, coefs, e0 = state["case"], state["dets"], state["coefs"], state["e0"]
    if kind == "sweep":
        d = state["pt2"].eval(dets, coefs, e0, case["k"], per_generator=case["host"])
        out = _totals(d)
        if case["k"]:
            out.update((f, _array(d[f])) for f in ("sel_dets", "sel_e", "sel_num"))
        if case["host"]:
            out.update((f, d[f]) for f in ("eps_by_rank", "na_by_rank", "ncon_by_rank", "rank_of"))
        return out
    if kind == "gens":
        d = state["pt2"].eval_generators(dets, coefs, e0, state["ranks"])
        return {f: d[f] for f in ("e_pt2", "sum_e_over_d", "n_perturbers", "n_connections", "eps", "s2", "na", "ncon")}
    if kind == "grad":
        de0, res = qp.qp_pt2_grad(state["pt2"].ctx, len(dets), dets, coefs, e0, state["dh"], state["deri"])
        return dict(_totals(res.as_dict()), dh=state["dh"], deri=state["deri"], de0=de0)
    if kind == "states":
        d = state["pt2"].eval_states(dets, coefs, e0, case["k"])
        return {f: d[f] for f in ("e_pt2_states", "sum_e_over_d_states", "n_perturbers", "n_connections", "min_abs_den",
                                  "sel_dets", "sel_crit", "sel_num")}
    if kind == "davidson":
        e, c, _ = state["pt2"].davidson(dets)
        return dict(e0=e, coefs=c)
    _, res = qp.qp_pt2_eval_noalloc(case["norb"], case["na"], case["nb"], state["h"], state["eri"], len(dets), dets, coefs,
                                    e0, case["k"], state["sel"], state["se"])
    m = res.n_selected
    return dict(_totals(res.as_dict()), sel_dets=state["sel"][:m], sel_e=state["se"][:m])


def work(case):
    """Bytes: integrals, determinants and coefficients read once, selections
    (or gradients, vectors) written once.  Operations: a multiply-add for each
    connection (J, alpha), of which there are N_det substitutions each, and
    for each perturber (about 0.4 per connection on such spaces) the diagonal,
    a reciprocal and three multiply-adds."""
    if case["kind"] == "batch":
        parts = [work(dict(c, kind="sweep")) for c in _batch_sizes(case)]
        return {f: sum(p[f] for p in parts) for f in ("bytes", "flops")}
    norb, ndet, kind = case["norb"], case["ndet"], case["kind"]
    m = norb * (norb + 1) // 2
    nst, word = case.get("nst", 1), 16 * ((norb - 1) // 64 + 1)
    eri = 8 * (m * (m + 1) // 2)
    data = eri // (2 if case.get("mixed") else 1) + ndet * (word + 8 * nst) + case.get("k", 0) * (word + 16)
    conn = case.get("ngen", ndet) * substitutions(norb, case["na"], case["nb"])
    if kind == "davidson":  # the matrix formed once; its entries cannot number more than the pairs
        nnz = min(ndet * (ndet - 1), 600 * ndet)
        return {"bytes": data + 12 * nnz, "flops": 40 * 2 * nnz}
    flops = nst * (2 * conn + 13 * 0.4 * conn)
    if kind == "grad":
        data += eri
        flops *= 2
    return {"bytes": int(data), "flops": int(flops)}


# ---------------------------------------------------------------------------
# the same quantities in plain FP64 torch
# ---------------------------------------------------------------------------
class _Plain:
    """Every single and double substitution of the determinants (one word per
    spin), with its phase and matrix element <J|H|alpha>."""

    def __init__(self, case, h, eri, dets):
        self.norb, self.n = case["norb"], (case["na"], case["nb"])
        self.h, self.eri, self.dev = h, eri, h.device
        orb = torch.arange(self.norb, device=self.dev)
        self.words = dets.reshape(-1, 2)
        self.bit = torch.bitwise_left_shift(torch.ones_like(orb), orb)
        self.occ = [((self.words[:, s, None] >> orb) & 1) for s in range(2)]
        self.olist = [torch.argsort(1 - o, dim=1, stable=True)[:, :n] for o, n in zip(self.occ, self.n)]
        self.vlist = [torch.argsort(o, dim=1, stable=True)[:, : self.norb - n] for o, n in zip(self.occ, self.n)]
        self.below = [torch.cumsum(o, 1) - o for o in self.occ]

    def v(self, p, q, r, s):
        return self.eri[_pair(_pair(p, q), _pair(r, s))]

    def between(self, s, rows, p, q):
        """Occupied orbitals of spin s strictly between p and q."""
        lo, hi = torch.minimum(p, q), torch.maximum(p, q)
        b, o = self.below[s], self.occ[s]
        return b[rows, hi] - b[rows, lo] - o[rows, lo]

    def all(self, lo, hi):
        """(J index, alpha words, element) of every substitution of J in [lo, hi)."""
        rows0 = torch.arange(lo, hi, device=self.dev)
        out = []

        def emit(rows, shape, flips, val, par):
            w = self.words[rows].expand(shape + (2,)).clone()
            for s, x in flips:
                w[..., s] ^= x
            val = torch.where((par % 2) == 1, -val, val)
            out.append((rows.expand(shape).reshape(-1), w.reshape(-1, 2), val.expand(shape).reshape(-1)))

        for s in range(2):
            rows = rows0[:, None, None]
            i, a = self.olist[s][lo:hi, :, None], self.vlist[s][lo:hi, None, :]
            shape = torch.broadcast_shapes(i.shape, a.shape)
            val = self.h[i, a]
            for t in range(2):
                for j in range(self.n[t]):
                    q = self.olist[t][lo:hi, j][:, None, None]
                    val = val + self.v(i, a, q, q)
                    if t == s:
                        val = val - self.v(i, q, q, a)
            emit(rows, shape, [(s, self.bit[i] ^ self.bit[a])], val, self.between(s, rows, i, a))
            n, m = self.n[s], self.norb - self.n[s]
            if n > 1 and m > 1:
                x, y = torch.triu_indices(n, n, 1, device=self.dev)
                i, j = self.olist[s][lo:hi, x][:, :, None], self.olist[s][lo:hi, y][:, :, None]
                x, y = torch.triu_indices(m, m, 1, device=self.dev)
                a, b = self.vlist[s][lo:hi, x][:, None, :], self.vlist[s][lo:hi, y][:, None, :]
                shape = torch.broadcast_shapes(i.shape, a.shape)
                inside = lambda z: ((z > torch.minimum(j, b)) & (z < torch.maximum(j, b))).long()
                par = self.between(s, rows, i, a) + self.between(s, rows, j, b) - inside(i) + inside(a)
                emit(rows, shape, [(s, self.bit[i] ^ self.bit[a] ^ self.bit[j] ^ self.bit[b])],
                     self.v(i, a, j, b) - self.v(i, b, j, a), par)
        rows = rows0[:, None, None, None, None]
        i, j = self.olist[0][lo:hi, :, None, None, None], self.olist[1][lo:hi, None, :, None, None]
        a, b = self.vlist[0][lo:hi, None, None, :, None], self.vlist[1][lo:hi, None, None, None, :]
        shape = torch.broadcast_shapes(i.shape, j.shape, a.shape, b.shape)
        par = self.between(0, rows, i, a) + self.between(1, rows, j, b)
        emit(rows, shape, [(0, self.bit[i] ^ self.bit[a]), (1, self.bit[j] ^ self.bit[b])], self.v(i, a, j, b), par)
        return tuple(torch.cat(x) for x in zip(*out))

    def diagonal(self, words):
        orb = torch.arange(self.norb, device=self.dev)
        J = self.v(orb[:, None], orb[:, None], orb[None, :], orb[None, :])
        K = self.v(orb[:, None], orb[None, :], orb[None, :], orb[:, None])
        out = []
        for w in words.split(1 << 20):
            n = [((w[:, s, None] >> orb) & 1).double() for s in range(2)]
            t = n[0] + n[1]
            e = t @ torch.diag(self.h) + 0.5 * ((t @ J) * t).sum(1)
            out.append(e - 0.5 * sum(((x @ K) * x).sum(1) for x in n))
        return torch.cat(out)


def _groups(plain):
    """Substitutions grouped by determinant: (J of each pair, element, group of
    each pair, words of each group), without the internal determinants."""
    n = len(plain.words)
    step = max(1, 20_000_000 // substitutions(plain.norb, *plain.n))
    parts = [plain.all(i, min(n, i + step)) for i in range(0, n, step)]
    J, words, val = (torch.cat(x) for x in zip(*parts))
    del parts
    key, inner = _mixed_key(words), torch.sort(_mixed_key(plain.words)).values
    pos = torch.searchsorted(inner, key).clamp(max=n - 1)
    ext = inner[pos] != key
    J, words, val, key = J[ext], words[ext], val[ext], key[ext]
    uniq, inv = torch.unique(key, return_inverse=True)
    g = torch.zeros((len(uniq), 2), dtype=torch.int64, device=key.device)
    g[inv] = words
    return J, val, inv, g


def _exact_sweep(case, plain, coefs, e0, per_generator=False):
    J, val, inv, words = _groups(plain)
    A = torch.zeros(len(words), dtype=torch.float64, device=val.device).index_add(0, inv, coefs[J] * val)
    D = e0 - plain.diagonal(words)
    e = A * A / D
    s2 = float((A / D).square().sum())
    out = dict(e_pt2=float(e.sum()), sum_e_over_d=s2, min_abs_den=float(D.abs().min()), z=1.0 / (1.0 + s2))
    out["e_rpt2"] = float(e0) + out["z"] * out["e_pt2"]
    if case["k"]:
        top = torch.sort(e.abs(), descending=True, stable=True).indices[: case["k"]]
        out.update(sel_e=e[top], sel_num=A[top])
    if per_generator:
        order = torch.sort(coefs * coefs, descending=True, stable=True).indices
        rank = torch.empty_like(order)
        rank[order] = torch.arange(len(order), device=order.device)
        gen = torch.full((len(words),), len(order), device=order.device).scatter_reduce(0, inv, rank[J], "amin")
        out["eps_by_rank"] = torch.zeros(len(order), dtype=torch.float64, device=e.device).index_add(0, gen, e)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "gens") or case["norb"] > 64 or case.get("mixed"):
        return None
    pairs = case["ndet"] * substitutions(case["norb"], case["na"], case["nb"])
    if pairs > (6.0e7 if kind == "grad" else 2.6e8) and kind != "davidson" or kind == "davidson" and (case["ndet"] > 1500 or pairs > 6e8):
        return None
    h, _, eri, dets, coefs, e0 = _instance(case, seed, case.get("nst", 1))
    if kind == "davidson":
        plain = _Plain(case, h, eri, dets)
        n = len(dets)
        H = torch.diag(plain.diagonal(plain.words))
        key = torch.sort(_mixed_key(plain.words))
        step = max(1, 20_000_000 // substitutions(plain.norb, *plain.n))
        for i in range(0, n, step):
            J, words, val = plain.all(i, min(n, i + step))
            k = _mixed_key(words)
            pos = torch.searchsorted(key.values, k).clamp(max=n - 1)
            hit = key.values[pos] == k
            H[J[hit], key.indices[pos[hit]]] = val[hit]
        ev, vec = torch.linalg.eigh(H)
        c = vec[:, 0] * (-1.0 if vec[0, 0] < 0 else 1.0)
        return dict(e0=float(ev[0]), coefs=c)
    if kind == "grad":
        h, eri = h.clone().requires_grad_(), eri.clone().requires_grad_()
        plain = _Plain(case, h, eri, dets)
        J, val, inv, words = _groups(plain)
        A = torch.zeros(len(words), dtype=torch.float64, device=val.device).index_add(0, inv, coefs[J] * val)
        D = e0 - plain.diagonal(words)
        E = (A * A / D).sum()
        gh, ge = torch.autograd.grad(E, [h, eri])
        A, D = A.detach(), D.detach()
        return dict(e_pt2=float(E.detach()), dh=0.5 * (gh + gh.T), deri=ge, de0=float(-(A / D).square().sum()))
    plain = _Plain(case, h, eri, dets)
    if kind == "states":
        J, val, inv, words = _groups(plain)
        H = plain.diagonal(words)
        e2, s2, crit = [], [], 0.0
        for s in range(case["nst"]):
            A = torch.zeros(len(words), dtype=torch.float64, device=val.device).index_add(0, inv, coefs[s][J] * val)
            D = (e0 - 0.2 * s) - H
            e2.append(float((A * A / D).sum()))
            s2.append(float((A / D).square().sum()))
            crit = crit + A * A / D / coefs[s].square().max()
            if s == 0:
                A0 = A
        top = torch.sort(crit.abs(), descending=True, stable=True).indices[: case["k"]]
        return dict(e_pt2_states=np.array(e2), sum_e_over_d_states=np.array(s2), sel_crit=crit[top], sel_num=A0[top])
    out = _exact_sweep(case, plain, coefs, e0, kind == "sweep" and case["host"])
    if kind == "noalloc":
        out.pop("sel_num", None)
    return out
