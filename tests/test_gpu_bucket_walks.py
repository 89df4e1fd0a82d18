"""The batched sigma and the density matrices at the (N-2) bucket sizes where their walks
change: the density matrices take buckets of 2 to 4 members in registers, up to 64 sorted and
larger ones in passes of 128 members; the batched sigma passes of 192 members.

One alpha and one beta electron share the empty (N-2) string, so a list of s such determinants
is one bucket of s members.  Every sum has at most s terms of one sign of rounding each, far
inside the bounds used (1e-11 relative for sigma, 1e-12 absolute for density matrices of a
normalised vector: the bounds of the other tests of these calls).
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_2501_18185_gb300 import sci
from paper_2501_18185_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _one_bucket(n, s, nvec=1):
    rng = np.random.default_rng(900 + s)
    ints = W.real_integrals(rng, n, 6, None)
    keys = np.sort(rng.choice(W.fci_keys(n, 1, 1), s, replace=False))
    return W.Workload(f"bucket_{s}", "spin_orbitals", n, 1, 1, keys, ints, rng.normal(size=(s, nvec)))


def test_batch_bucket_sizes(gpu):
    torch = gpu
    ws = [_one_bucket(22, s) for s in (2, 31, 32, 33, 191, 192, 193, 384, 385, 484)]
    ws.append(W.random_small(73, "spin_orbitals", 9, 2, 2, frac=0.3))
    B = sci.Batch([sci.Hamiltonian.from_workload(w) for w in ws])
    C = torch.from_numpy(np.concatenate([w.c[:, 0] for w in ws])).cuda()
    B.plan(sci.SCI_SCHED_TILE, C, torch.empty_like(C))
    S = B.sigma(C).cpu().numpy()
    for w, off in zip(ws, B.offsets):
        ref = Oracle.from_workload(w).sigma(w.c)[:, 0]
        assert np.linalg.norm(S[off:off + w.M] - ref) <= 1e-11 * np.linalg.norm(ref), w.name


@pytest.mark.parametrize("s", [2, 3, 4, 5, 6, 32, 33, 63, 64, 65, 66, 256, 257, 258, 484])
@pytest.mark.parametrize("nvec", [1, 3, 9])
def test_rdm_bucket_sizes(gpu, s, nvec):
    torch = gpu
    w = _one_bucket(22, s, nvec)
    C = w.c / np.linalg.norm(w.c, axis=0)
    weights = np.linspace(1.0, 0.2, nvec) / nvec
    H = sci.Hamiltonian.from_workload(w)
    g1, g2 = H.rdm12(torch.from_numpy(C).cuda(), weights=weights)
    o = Oracle.from_workload(w)
    r1 = r2 = 0.0
    for k in range(nvec):
        a, b = o.rdm12(np.ascontiguousarray(C[:, k]))
        r1, r2 = r1 + weights[k] * a, r2 + weights[k] * b
    assert np.abs(g1.cpu().numpy() - r1).max() < 1e-12
    assert np.abs(g2.cpu().numpy() - r2).max() < 1e-12


@pytest.mark.parametrize("frac", [0.06, 0.5])
def test_rdm_mixed_buckets_complex(gpu, frac):
    torch = gpu
    w = W.random_small(71, "spinors", 14, 4, 0, frac=frac, nvec=2)
    C = w.c / np.linalg.norm(w.c, axis=0)
    H = sci.Hamiltonian.from_workload(w)
    g1, g2 = H.rdm12(torch.from_numpy(C).cuda(), weights=[0.75, -0.25])
    o = Oracle.from_workload(w)
    refs = [o.rdm12(np.ascontiguousarray(C[:, k])) for k in range(2)]
    for got, k in ((g1, 0), (g2, 1)):
        assert np.abs(got.cpu().numpy() - (0.75 * refs[0][k] - 0.25 * refs[1][k])).max() < 1e-12
