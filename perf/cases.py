"""The work this framework is measured on, one public call (or one forward and backward) a case.

Each case names an operation and a determinant space:

  sigma          S = H C by Hamiltonian.sigma, C of one or more vectors, in FP64, paired
                 FP32 ("ds") or FP32 storage ("f32")
  rdm12          one- and two-particle density matrices of a weighted set of vectors
  energy         forward and backward of the differentiable Rayleigh quotients
  batch          S = H_i C_i of many small full-CI instances in one launch
  determinants   loading a determinant list: validation, connection tables, diagonal
  enpt2          second-order energies of the external space

  fci            every determinant of n orbitals, na + nb electrons
  sel            selected spin-orbital space, HF + singles + doubles + random triples and
                 quadruples, one-word strings
  words          the same with random triples only, strings of two to four words
  spinor         selected spinor space (complex), HF + singles + doubles + random triples
"""
import math
from math import comb

import numpy as np
import torch

from paper_2501_18185_gb300 import sci
from paper_2501_18185_gb300 import workloads as W
from paper_2501_18185_gb300.autograd import rayleigh_energy

_PREC = {"f64": sci.SCI_PREC_F64, "ds": sci.SCI_PREC_F64_DS, "f32": sci.SCI_PREC_F32_STORE_F64_ACC}


def listed():
    return [
        {"name": "sigma_fci_8o", "op": "sigma", "space": "fci", "n": 8, "na": 4, "nb": 4, "nvec": 1, "prec": "f64"},
        {"name": "sigma_30o_60k", "op": "sigma", "space": "sel", "n": 30, "na": 10, "nb": 10, "M": 60_000, "nvec": 1,
         "prec": "f64"},
        {"name": "sigma_30o_2m", "op": "sigma", "space": "sel", "n": 30, "na": 10, "nb": 10, "M": 2_000_000, "nvec": 1,
         "prec": "f64"},
        {"name": "sigma_30o_f32_x8", "op": "sigma", "space": "sel", "n": 30, "na": 10, "nb": 10, "M": 500_000,
         "nvec": 8, "prec": "f32"},
        {"name": "sigma_27o_ds_x3", "op": "sigma", "space": "sel", "n": 27, "na": 9, "nb": 8, "M": 300_001, "nvec": 3,
         "prec": "ds"},
        {"name": "sigma_64s", "op": "sigma", "space": "spinor", "n": 64, "na": 14, "nb": -1, "M": 500_001, "nvec": 1,
         "prec": "f64"},
        {"name": "sigma_40o_x2", "op": "sigma", "space": "words", "n": 40, "na": 4, "nb": 4, "M": 400_000, "nvec": 2,
         "prec": "f64"},
        {"name": "rdm12_30o_x4", "op": "rdm12", "space": "sel", "n": 30, "na": 10, "nb": 10, "M": 250_000, "nvec": 4},
        {"name": "energy_30o_x4", "op": "energy", "space": "sel", "n": 30, "na": 10, "nb": 10, "M": 100_000, "nvec": 4},
        {"name": "batch_fci_x32", "op": "batch", "space": "fci", "count": 32, "max_dim": 100_000},
        {"name": "determinants_30o", "op": "determinants", "space": "sel", "n": 30, "na": 10, "nb": 10, "M": 400_000},
        {"name": "enpt2_24o_x2", "op": "enpt2", "space": "sel", "n": 24, "na": 6, "nb": 6, "M": 40_000, "nvec": 2},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(case)["flops"] for case in listed())
    while True:
        case = _draw(rng)
        if work(case)["flops"] <= most:
            return case


def _draw(rng):
    op = rng.choice(["sigma"] * 6 + ["rdm12", "energy", "batch", "determinants", "enpt2"])
    if op == "batch":
        return {"op": op, "space": "fci", "count": rng.randint(3, 40), "max_dim": _log_uniform(rng, 2_000, 80_000)}
    space = rng.choice(["fci", "sel", "sel", "words", "spinor"]) if op == "sigma" else "sel"
    case = {"op": op, "space": space}
    if space == "fci":
        case.update(n=rng.randint(6, 10), na=rng.randint(2, 5), nb=rng.randint(2, 5))
    elif space == "spinor":
        case.update(n=rng.randint(40, 64), na=rng.randint(8, 14), nb=-1)
    elif space == "words":
        case.update(n=rng.choice([rng.randint(34, 60), rng.randint(66, 72)]), na=rng.randint(2, 4), nb=rng.randint(2, 3))
    elif op == "enpt2":
        case.update(n=rng.randint(18, 24), na=rng.randint(4, 6), nb=rng.randint(4, 6))
    else:
        case.update(n=rng.randint(22, 30), na=rng.randint(6, 10), nb=rng.randint(6, 10))
    if space != "fci":
        # from just above HF + singles + doubles to the top of the range of the operation
        sizes = _level_sizes(case)
        lo = sum(sizes[:3])
        top = {"sigma": 800_000, "rdm12": 300_000, "energy": 150_000, "determinants": 500_000, "enpt2": 40_000}[op]
        case["M"] = _log_uniform(rng, lo, min(max(top, lo + 1), lo + sizes[3] // 2))
    if op == "sigma":
        case["nvec"] = rng.choice([1, 1, 2, 3, 4, 8])
        case["prec"] = rng.choice(["f64", "f64", "ds"] if space == "spinor" else ["f64", "f64", "ds", "f32"])
        if space == "spinor":
            case["nvec"] = min(case["nvec"], 2)
    elif op != "determinants":
        case["nvec"] = rng.randint(1, 4)
    return case


# ------------------------------------------------------------------ inputs
def _level_sizes(case):
    """Determinants at excitation level 0..4 from the reference."""
    n, na, nb = case["n"], case["na"], case["nb"]
    one = [W.n_strings_at_level(n, na, k) for k in range(5)]
    if case["space"] == "spinor":
        return one
    two = [W.n_strings_at_level(n, nb, k) for k in range(5)]
    return [sum(one[k] * two[level - k] for k in range(level + 1)) for level in range(5)]


def _workload(case, seed):
    """Integrals, sorted determinant list and vectors of a case."""
    n, na, nb, nvec = case["n"], case["na"], case["nb"], case.get("nvec", 1)
    rng = np.random.default_rng([seed, 97])
    if case["space"] == "fci":
        ints = W.real_integrals(rng, n, 2 * n, None)
        keys = W.fci_keys(n, na, nb)
        w = W.Workload("fci", "spin_orbitals", n, na, nb, keys, ints, None)
        w.c = W.coefficient_vector(rng, keys, w.hf_key(), nvec, decay_by_level=False)
        return w
    if case["space"] == "words":
        words = -(-2 * n // 64)
        return W.selected_words(n, na, nb, case["M"], words, naux=40, nvec=nvec, seed=[seed, 98])
    if case["space"] == "spinor":
        ints = W.complex_integrals(rng, n, 80, 0.95)
        keys, _ = W.selected_spinor_keys(rng, n, na, case["M"])
        w = W.Workload("spinor", "spinors", n, na, -1, keys, ints, None)
    else:
        ints = W.real_integrals(rng, n, 4 * n, 0.95)
        keys, _ = W.selected_spin_orbital_keys(rng, n, na, nb, case["M"])
        w = W.Workload("sel", "spin_orbitals", n, na, nb, keys, ints, None)
    w.c = W.coefficient_vector(rng, keys, w.hf_key(), nvec, ints.complex_)
    return w


def _instances(case, seed):
    """The small full-CI instances of a batch."""
    rng = np.random.default_rng([seed, 99])
    shapes = np.random.default_rng(case["count"])      # the shapes belong to the case
    out = []
    while len(out) < case["count"]:
        n, na, nb = int(shapes.integers(6, 15)), int(shapes.integers(2, 8)), int(shapes.integers(2, 8))
        if na > n or nb > n or comb(n, na) * comb(n, nb) > case["max_dim"]:
            continue
        keys = W.fci_keys(n, na, nb)
        ints = W.real_integrals(rng, n, n, None)
        c = W.coefficient_vector(rng, keys, np.uint64(0), 1, decay_by_level=False)
        out.append(W.Workload(f"i{len(out)}", "spin_orbitals", n, na, nb, keys, ints, c))
    return out


def _weights(nvec):
    return np.arange(nvec, 0, -1) / (nvec * (nvec + 1) / 2)


def _device_vectors(case, w):
    return torch.from_numpy(w.c).cuda().to(torch.float32 if case.get("prec") == "f32" else torch.from_numpy(w.c).dtype)


def prepare(case, seed):
    if case["op"] == "batch":
        ws = _instances(case, seed)
        batch = sci.Batch([sci.Hamiltonian.from_workload(w) for w in ws])
        batch.plan()
        return {"op": "batch", "batch": batch, "C": torch.from_numpy(np.concatenate([w.c[:, 0] for w in ws])).cuda()}
    w = _workload(case, seed)
    state = {"op": case["op"], "C": _device_vectors(case, w)}
    if case["op"] == "determinants":
        H = sci.Hamiltonian()
        H.set_integrals(w.mode, w.ints.h, chol=w.ints.chol)
        state.update(H=H, keys=torch.from_numpy(w.keys.view(np.int64)).cuda(), na=w.n_alpha, nb=w.n_beta)
        return state
    state["H"] = sci.Hamiltonian.from_workload(w)
    if case["op"] == "sigma":
        state["prec"] = _PREC[case["prec"]]
    elif case["op"] == "rdm12":
        state["weights"] = _weights(case["nvec"])
    elif case["op"] == "energy":
        state["h"] = torch.from_numpy(w.ints.h).cuda().requires_grad_(True)
        state["L"] = torch.from_numpy(w.ints.chol).cuda().requires_grad_(True)
        state["C"].requires_grad_(True)
        state["weights"] = torch.from_numpy(_weights(case["nvec"])).cuda()
    elif case["op"] == "enpt2":
        state["E0"] = w.ints.h.trace() - 50.0 - np.arange(case["nvec"])
    return state


def run(state):
    op = state["op"]
    if op == "batch":
        return state["batch"].sigma(state["C"])
    H = state["H"]
    if op == "sigma":
        return H.sigma(state["C"], prec=state["prec"])
    if op == "rdm12":
        return H.rdm12(state["C"], weights=state["weights"])
    if op == "energy":
        E = rayleigh_energy(state["h"], state["L"], state["C"], H)
        gh, gL, gC = torch.autograd.grad(E, (state["h"], state["L"], state["C"]), state["weights"])
        return {"E": E.detach(), "gh": gh, "gL": gL, "gC": gC}
    if op == "determinants":
        H.set_determinants(state["keys"], state["na"], state["nb"])
        return {"diagonal": H.diagonal(), "pairs": H.count_pairs()}
    e2w, e2p, e2q, _ = H.enpt2(state["C"], state["E0"])
    return {"E2W": e2w, "E2P": e2p, "E2Q": e2q}


# ------------------------------------------------------------------ the work of a case
def _moves(n, nocc, k):
    """{change of k: count} of the single and of the double excitations, within one spin,
    of a string with k holes in the reference."""
    o, v = nocc - k, n - nocc - k
    single = {1: o * v, 0: o * k + k * v, -1: k * k}
    double = {}
    for r in range(3):          # electrons taken from reference orbitals
        for s in range(3):      # electrons put into holes of the reference
            cnt = comb(max(o, 0), r) * comb(k, 2 - r) * comb(k, s) * comb(max(v, 0), 2 - s)
            double[r - s] = double.get(r - s, 0) + cnt
    return single, double


def _pairs(case):
    """Connected ordered pairs (I, J), I != J, of the case's space: exact for a full CI,
    the expectation for spaces with randomly drawn levels."""
    n, na, nb = case["n"], case["na"], case["nb"]
    spinor = case["space"] == "spinor"
    sizes = _level_sizes(case)
    if case["space"] == "fci":
        M = comb(n, na) * comb(n, nb)
        sa, sb = na * (n - na), nb * (n - nb)
        return M * (sa + sb + sa * sb + comb(na, 2) * comb(n - na, 2) + comb(nb, 2) * comb(n - nb, 2))
    rest = case["M"] - sum(sizes[:3])
    fill = [1.0, 1.0, 1.0, 0.0, 0.0]
    if case["space"] == "sel":
        fill[3], fill[4] = ((rest + 1) // 2) / max(sizes[3], 1), (rest // 2) / max(sizes[4], 1)
    else:
        fill[3] = rest / max(sizes[3], 1)

    def at(level):
        return fill[level] if 0 <= level < 5 else 0.0

    total = 0.0
    for ka in range(5):
        for kb in range(1 if spinor else 5 - ka):
            count = W.n_strings_at_level(n, na, ka) * (1 if spinor else W.n_strings_at_level(n, nb, kb))
            if count == 0 or at(ka + kb) == 0.0:
                continue
            s1, d1 = _moves(n, na, ka)
            neighbours = sum(c * at(ka + kb + d) for m in (s1, d1) for d, c in m.items())
            if not spinor:
                s2, d2 = _moves(n, nb, kb)
                neighbours += sum(c * at(ka + kb + d) for m in (s2, d2) for d, c in m.items())
                neighbours += sum(x * y * at(ka + kb + d + e) for d, x in s1.items() for e, y in s2.items())
            total += count * at(ka + kb) * neighbours
    return total


def _size(case):
    return comb(case["n"], case["na"]) * comb(case["n"], case["nb"]) if case["space"] == "fci" else case["M"]


def work(case):
    op = case["op"]
    if op == "batch":
        by, fl = 0, 0
        for w in _instances(case, 0):
            sub = {"space": "fci", "n": w.n, "na": w.n_alpha, "nb": w.n_beta}
            by += 8 * (3 * w.M + w.n ** 2 + w.n ** 3)
            fl += 2 * (_pairs(sub) + w.M)
        return {"bytes": by, "flops": fl}
    n, M, nvec = case["n"], _size(case), case.get("nvec", 1)
    spinor = case["space"] == "spinor"
    words = 1 if spinor else -(-2 * n // 64)
    naux = {"fci": 2 * n, "sel": 4 * n, "words": 40, "spinor": 80}[case["space"]]
    scalar = 16 if spinor else 8
    inputs = 8 * words * M + scalar * (naux + 1) * n * n      # the strings and the integrals
    if op == "determinants":
        N = case["na"] + case["nb"]
        return {"bytes": 8 * words * M + 8 * M, "flops": M * N * N}
    pairs = _pairs(case) + M
    if op == "sigma":
        c = 4 if case["prec"] == "f32" else scalar
        return {"bytes": inputs + M * nvec * (c + scalar), "flops": (8 if spinor else 2) * nvec * pairs}
    if op == "rdm12":
        return {"bytes": 8 * words * M + 8 * M * nvec + 8 * ((2 * n) ** 2 + (2 * n) ** 4), "flops": 2 * nvec * pairs}
    if op == "energy":
        return {"bytes": 2 * inputs + 3 * 8 * M * nvec, "flops": 4 * nvec * pairs + 4 * naux * n ** 4}
    N, virt = case["na"] + case["nb"], 2 * n - case["na"] - case["nb"]      # enpt2
    s, d = _moves(n, case["na"], 0), _moves(n, case["nb"], 0)
    moves = sum(s[0].values()) + sum(d[0].values()) + sum(s[1].values()) + sum(d[1].values())
    moves += sum(s[0].values()) * sum(d[0].values())
    assert moves <= comb(N, 2) * comb(virt, 2) + N * virt
    return {"bytes": inputs + 8 * M * nvec, "flops": 2 * nvec * moves * M}


# ------------------------------------------------------------------ 64-bit values
# The same quantities from the occupation numbers, in torch's float64 / complex128: pairs
# of determinants by the number of orbitals they share, elements by the Slater-Condon rules.
class _Exact:
    def __init__(self, w):
        dev = "cuda"
        keys = w.keys if w.keys.ndim == 2 else w.keys[:, None]
        self.norb = w.n if w.mode == "spinors" else 2 * w.n
        bits = [(keys[:, p // 64] >> np.uint64(p % 64)) & np.uint64(1) for p in range(self.norb)]
        self.occ = torch.from_numpy(np.stack(bits, axis=1).astype(np.int8)).to(dev)
        self.M, self.N = self.occ.shape[0], int(self.occ[0].sum())
        self.below = torch.cumsum(self.occ, 1, dtype=torch.int32) - self.occ
        h = torch.from_numpy(w.ints.h).to(dev)
        L = torch.from_numpy(w.ints.chol).to(dev)
        naux, n = L.shape[0], w.n
        eri = (L.reshape(naux, -1).T @ L.reshape(naux, -1)).reshape(n, n, n, n)
        self.n, self.h, self.eri, self.L = n, h, eri, L
        p = torch.arange(self.norb, device=dev)
        self.orb = p % n if w.mode != "spinors" else p
        self.spin = p // n if w.mode != "spinors" else torch.zeros_like(p)
        o, same = self.orb, (self.spin[:, None] == self.spin[None, :])
        self.h_so = h[o][:, o] * same
        coul = torch.einsum("aikk->aik", eri)[o][:, o][:, :, o] * same[:, :, None]
        exch = torch.einsum("akki->aik", eri)[o][:, o][:, :, o] * (same[:, None, :] & same[None, :, :])
        self.g = coul - exch                      # [a, i, k] = (ai|kk) - (ak|ki)
        hd = torch.diagonal(self.h_so).real
        jk = torch.einsum("iik->ik", self.g).real
        x = self.occ.to(torch.float64)
        self.diag = x @ hd + 0.5 * ((x @ jk) * x).sum(1)

    def two(self, a, i, b, j):
        """(ai|bj) over spin-orbitals"""
        v = self.eri[self.orb[a], self.orb[i], self.orb[b], self.orb[j]]
        return v * ((self.spin[a] == self.spin[i]) & (self.spin[b] == self.spin[j]))

    def pairs(self, chunk=1 << 30, most=1 << 23):
        """(I, J, degree) of the connected pairs, in blocks of one degree each"""
        occ = self.occ.to(torch.float16)
        rows = max(1, chunk // max(self.M, 1))
        for r in range(0, self.M, rows):
            common = occ[r:r + rows] @ occ.T
            for degree in (1, 2):
                I, J = torch.nonzero(common == self.N - degree, as_tuple=True)
                for t in range(0, len(I), most):
                    yield I[t:t + most] + r, J[t:t + most], degree

    def excitation(self, I, J, degree):
        """sign, and the orbitals i.. of J and a.. of I that differ, ascending"""
        d = self.occ[I] - self.occ[J]
        last = self.norb - 1
        created = [(d == 1).to(torch.int8).argmax(1)]
        taken = [(d == -1).to(torch.int8).argmax(1)]
        if degree == 2:
            created.append(last - (d.flip(1) == 1).to(torch.int8).argmax(1))
            taken.append(last - (d.flip(1) == -1).to(torch.int8).argmax(1))
        cnt = self.below[J]
        parity = torch.zeros_like(I)
        for x in created + taken:       # electrons below x, the taken ones left out
            parity += cnt.gather(1, x[:, None])[:, 0]
            for t in taken:
                parity -= (t < x).to(parity.dtype)
        return 1.0 - 2.0 * (parity & 1).to(torch.float64), taken, created

    def elements(self, I, J, degree, move):
        sign, taken, created = move
        if degree == 1:
            a, i = created[0], taken[0]
            return sign * (self.h_so[a, i] + (self.g[a, i] * self.occ[J].to(torch.float64)).sum(1))
        (i, j), (a, b) = taken, created
        return sign * (self.two(a, i, b, j) - self.two(a, j, b, i))

    def sigma(self, C):
        S = self.diag[:, None] * C
        for I, J, degree in self.pairs():
            v = self.elements(I, J, degree, self.excitation(I, J, degree))
            for k in range(C.shape[1]):
                S[:, k].index_add_(0, I, v * C[J, k])
        return S

    def rdm(self, C, weights):
        no, x = self.norb, self.occ.to(torch.float64)
        w = torch.as_tensor(weights, device=C.device)
        g1 = torch.zeros((no, no), dtype=C.dtype, device=C.device)
        g2 = torch.zeros(no ** 4, dtype=C.dtype, device=C.device)

        def add(p, q, r, s, v):        # <a+_p a+_r a_s a_q>
            g2.index_add_(0, ((p * no + q) * no + r) * no + s, v)

        p2 = (C * C) @ w
        g1 += torch.diag((x * p2[:, None]).sum(0))
        both = (x * p2[:, None]).T @ x
        p, r = torch.nonzero(1 - torch.eye(no, device=C.device), as_tuple=True)
        add(p, p, r, r, both[p, r])
        add(p, r, r, p, -both[p, r])
        ks = torch.arange(no, device=C.device)
        for I, J, degree in self.pairs(most=1 << 21):
            sign, taken, created = self.excitation(I, J, degree)
            v = sign * ((C[I] * C[J]) @ w)
            if degree == 2:
                (i, j), (a, b) = taken, created
                add(a, i, b, j, v), add(b, j, a, i, v), add(a, j, b, i, -v), add(b, i, a, j, -v)
                continue
            a, i = created[0], taken[0]
            g1.view(-1).index_add_(0, a * no + i, v)
            both = (x[J] * x[I]) * v[:, None]
            a, i, k = a[:, None].expand_as(both), i[:, None].expand_as(both), ks.expand_as(both)
            a, i, k, u = (t.reshape(-1) for t in (a, i, k, both))
            add(a, i, k, k, u), add(k, k, a, i, u), add(a, k, k, i, -u), add(k, i, a, k, -u)
        return g1, g2.view(no, no, no, no)

    def enpt2(self, C, E0, block=512):
        """E2[W], E2[P], E2[Q] by generating every excitation of every determinant"""
        dev, no, nv = C.device, self.norb, C.shape[1]
        weight = torch.ones(no, dtype=torch.int64, device=dev) << torch.arange(no, device=dev)
        keys = (self.occ.to(torch.int64) * weight).sum(1)
        order = torch.arange(no, device=dev)
        N, V = self.N, no - self.N
        i2, j2 = (t.to(dev) for t in torch.triu_indices(N, N, 1))
        a2, b2 = (t.to(dev) for t in torch.triu_indices(V, V, 1))
        ks, vs = [], []

        def put(J, key, v):
            ks.append(key), vs.append(v[:, None] * C[J])

        for r in range(0, self.M, block):
            occ = self.occ[r:r + block].to(torch.int64)
            B = occ.shape[0]
            o = torch.argsort(1 - occ, dim=1, stable=True)[:, :N]
            v = torch.argsort(occ, dim=1, stable=True)[:, :V]
            cnt = self.below[r:r + block].to(torch.int64)
            rows = torch.arange(B, device=dev) + r
            # singles
            i, a = o[:, :, None].expand(B, N, V), v[:, None, :].expand(B, N, V)
            J = rows[:, None, None].expand(B, N, V)
            ok = self.spin[i] == self.spin[a]
            i, a, J = i[ok], a[ok], J[ok]
            par = cnt[J - r, i] + cnt[J - r, a] - (i < a).to(torch.int64)
            el = self.h_so[a, i] + (self.g[a, i] * self.occ[J].to(torch.float64)).sum(1)
            put(J, keys[J] - weight[i] + weight[a], el * (1 - 2 * (par & 1)))
            # doubles
            i, j = o[:, i2][:, :, None], o[:, j2][:, :, None]
            a, b = v[:, a2][:, None, :], v[:, b2][:, None, :]
            ok = self.spin[i] + self.spin[j] == self.spin[a] + self.spin[b]
            J, ij, ab = torch.nonzero(ok, as_tuple=True)
            i, j, a, b = o[J, i2[ij]], o[J, j2[ij]], v[J, a2[ab]], v[J, b2[ab]]
            par = torch.zeros_like(J)
            for x in (i, j, a, b):
                par += cnt[J, x] - (i < x).to(torch.int64) - (j < x).to(torch.int64)
            el = (self.two(a, i, b, j) - self.two(a, j, b, i)) * (1 - 2 * (par & 1))
            J = J + r
            put(J, keys[J] - weight[i] - weight[j] + weight[a] + weight[b], el)
        key, inv = torch.unique(torch.cat(ks), return_inverse=True)
        R = torch.zeros((len(key), nv), dtype=torch.float64, device=dev)
        R.index_add_(0, inv, torch.cat(vs))
        at = torch.searchsorted(key, keys)
        hit = key[at.clamp(max=len(key) - 1)] == keys
        inside = torch.where(hit[:, None], R[at.clamp(max=len(key) - 1)], 0.0)     # <I|H|c> - c_I H_II
        hd = torch.diagonal(self.h_so).real
        jk = torch.einsum("iik->ik", self.g).real
        W2 = torch.zeros(nv, dtype=torch.float64, device=dev)
        e0 = torch.as_tensor(np.asarray(E0), device=dev)
        for t in range(0, len(key), 1 << 22):
            x = ((key[t:t + (1 << 22), None] >> order) & 1).to(torch.float64)
            d = x @ hd + 0.5 * ((x @ jk) * x).sum(1)
            W2 += (R[t:t + (1 << 22)] ** 2 / (e0 - d[:, None])).sum(0)
        P2 = (inside ** 2 / (e0 - self.diag[:, None])).sum(0)
        return W2, P2, W2 - P2


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        parts = [(_Exact(w), torch.from_numpy(w.c).cuda()) for w in _instances(case, seed)]
        return torch.cat([x.sigma(c)[:, 0] for x, c in parts])
    words = -(-2 * case["n"] // 64)
    limit = {"sigma": 500_001, "rdm12": 250_000, "energy": 100_000, "determinants": 400_000, "enpt2": 40_000}[op]
    if _size(case) > limit or (case["space"] == "words" and words > 4):
        return None
    if op != "determinants" and _pairs(case) * case["nvec"] > 3e9:
        return None
    w = _workload(case, seed)
    x = _Exact(w)
    C = torch.from_numpy(w.c).cuda()
    if case.get("prec") == "f32":
        C = C.float().double()
    if op == "sigma":
        return x.sigma(C)
    if op == "determinants":
        return {"diagonal": x.diag, "pairs": None}
    if op == "rdm12":
        return x.rdm(C, _weights(case["nvec"]))
    if op == "enpt2":
        if x.M * work(case)["flops"] / (2 * case["nvec"] * x.M) > 7e8:
            return None
        E2 = x.enpt2(C, w.ints.h.trace() - 50.0 - np.arange(case["nvec"]))
        return dict(zip(("E2W", "E2P", "E2Q"), (t.cpu().numpy() for t in E2)))
    S, den = x.sigma(C), (C * C).sum(0)
    E = (C * S).sum(0) / den
    G = torch.from_numpy(_weights(case["nvec"])).cuda() / den
    g1, g2 = x.rdm(C, G.cpu().numpy())
    n = x.n
    gam2 = g2.view(2, n, 2, n, 2, n, 2, n)
    gam2 = torch.einsum("apaqbrbs->pqrs", gam2)
    gL = (gam2.reshape(n * n, n * n) @ x.L.reshape(-1, n * n).T).T.reshape(x.L.shape)
    return {"E": E, "gh": g1[:n, :n] + g1[n:, n:], "gL": gL, "gC": 2.0 * (S - C * E) * G}
