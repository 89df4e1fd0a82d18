"""Sigma where the choice of the double-excitation kernels changes with the space: a pair table
above the size that is taken as close to the SMs, where one FP64 vector walks 5 to 32 members
aligned and sorts 33 to 64, and lists of few and of many table entries, where the paired-FP32
and FP32-storage launches take one walk or walks by bucket size.

Every precision at one, two, three and eight vectors (four complex) equals the oracle on a sample of
rows (1e-11 of the row norms; FP32 storage row by row within the rounding of the pair table), over
the whole list, over a row range and in the deterministic mode.
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_2501_18185_gb300 import sci
from paper_2501_18185_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-11
U32 = 2.0 ** -24   # rounding of the FP32 pair table, the one rounding left when C is FP32


def _one_bucket(s):
    rng = np.random.default_rng(800 + s)
    ints = W.real_integrals(rng, 20, 6, None)      # a pair table of 1.9 MB
    keys = np.sort(rng.choice(W.fci_keys(20, 1, 1), s, replace=False))
    return W.Workload(f"bucket_{s}", "spin_orbitals", 20, 1, 1, keys, ints, rng.normal(size=(s, 8)))


def _selected(n, na, nb, M):
    rng = np.random.default_rng(n)
    ints = W.real_integrals(rng, n, 6, None)
    keys, _ = W.selected_spin_orbital_keys(rng, n, na, nb, M)
    return W.Workload("selected", "spin_orbitals", n, na, nb, keys, ints, rng.normal(size=(M, 8)))


SPACES = {f"bucket_{s}": (lambda s=s: _one_bucket(s)) for s in (4, 5, 31, 32, 33, 63, 64, 65)}
SPACES["all_sizes_few"] = lambda: _selected(19, 2, 2, 3000)
SPACES["all_sizes"] = lambda: _selected(20, 3, 3, 45000)
SPACES["all_sizes_small_table"] = lambda: _selected(12, 4, 4, 20000)
SPACES["up_to_49"] = lambda: W.random_small(75, "spin_orbitals", 10, 4, 4, frac=0.3, nvec=8)
SPACES["complex"] = lambda: W.random_small(77, "spinors", 20, 6, 0, frac=0.5, nvec=4)


def entries_by_size(w):
    """Entries of the (N-2) table in buckets of 2 to 4, 5 to 32, 33 to 64 and more members."""
    norb = w.n if w.mode == "spinors" else 2 * w.n
    occ = np.nonzero((w.keys[:, None] >> np.arange(norb, dtype=np.uint64)) & np.uint64(1))[1].reshape(w.M, -1)
    bit = np.uint64(1) << occ.astype(np.uint64)
    sub = [w.keys ^ bit[:, i] ^ bit[:, j] for i in range(occ.shape[1]) for j in range(i)]
    size = np.unique(np.concatenate(sub), return_counts=True)[1]
    return [int(size[(size >= lo) & (size <= hi)].sum()) for lo, hi in ((2, 4), (5, 32), (33, 64), (65, 1 << 30))]


@pytest.mark.parametrize("name", list(SPACES))
def test_dispatch(gpu, name):
    torch = gpu
    w = SPACES[name]()
    parts = entries_by_size(w)
    if name.startswith("all_sizes"):
        assert min(parts) > 0
    if w.M > 10000:
        assert sum(parts[:3]) > 200_000
    o = Oracle.from_workload(w)
    H = sci.Hamiltonian.from_workload(w)
    cplx = np.iscomplexobj(w.c)
    rows = np.unique(np.random.default_rng(1).integers(0, w.M, 150))
    a, b = w.M // 3, w.M - w.M // 4
    for prec in [sci.SCI_PREC_F64, sci.SCI_PREC_F64_DS] + ([] if cplx else [sci.SCI_PREC_F32_STORE_F64_ACC]):
        f32 = prec == sci.SCI_PREC_F32_STORE_F64_ACC
        for nvec in (1, 2, 3, 4) if cplx else (1, 2, 3, 8):
            t = torch.from_numpy(np.ascontiguousarray(w.c[:, :nvec])).cuda()
            t = t.float() if f32 else t
            C = t.double().cpu().numpy() if f32 else t.cpu().numpy()
            S = H.sigma(t, prec=prec).cpu().numpy()
            ref = o.sigma_rows(rows, C).reshape(len(rows), nvec)
            if f32:
                A = o.sigma_abs_rows(rows, C).reshape(len(rows), nvec)
                assert (np.abs(S[rows] - ref) <= 1.05 * U32 * A + 1e-300).all()
            else:
                assert np.linalg.norm(S[rows] - ref) <= TOL * np.linalg.norm(ref)
            part = torch.full((w.M, nvec), 7.0, dtype=torch.complex128 if cplx else torch.float64, device="cuda")
            H.set_row_range(a, b)
            H.sigma(t, out=part, prec=prec)
            H.set_row_range(0, w.M)
            part = part.cpu().numpy()
            assert np.abs(part[a:b] - S[a:b]).max() <= 1e-13 * np.abs(S).max()
            assert (part[:a] == 7.0).all() and (part[b:] == 7.0).all()
            H.set_deterministic(nvec)
            D1, D2 = H.sigma(t, prec=prec).cpu().numpy(), H.sigma(t, prec=prec).cpu().numpy()
            H.set_deterministic(0)
            assert np.array_equal(D1, D2)
            assert np.abs(D1 - S).max() <= 1e-13 * np.abs(S).max()


def test_short_ranges(gpu):
    """Row ranges of a few rows, whose tables in FP32 storage take one walk where the whole list
    goes by size, and of most rows."""
    torch = gpu
    w = SPACES["all_sizes"]()
    H = sci.Hamiltonian.from_workload(w)
    for nvec in (1, 3, 8):
        t = torch.from_numpy(np.ascontiguousarray(w.c[:, :nvec])).cuda().float()
        S = H.sigma(t, prec=sci.SCI_PREC_F32_STORE_F64_ACC)
        for a, b in ((0, 1), (w.M // 2, w.M // 2 + 64), (w.M - 5000, w.M), (1, w.M)):
            part = torch.full((w.M, nvec), 7.0, dtype=torch.float64, device="cuda")
            H.set_row_range(a, b)
            H.sigma(t, out=part, prec=sci.SCI_PREC_F32_STORE_F64_ACC)
            H.set_row_range(0, w.M)
            assert (part[a:b] - S[a:b]).abs().max() <= 1e-13 * S.abs().max()
            assert (part[:a] == 7.0).all() and (part[b:] == 7.0).all()
