"""ENPT2 of determinants far from the lowest-orbital reference (more than 32 orbitals differ,
past the list of the evaluation kernel) against the same space with the orbitals numbered
backwards, where they are the reference and its excitations.  Reversing the orbitals multiplies
every determinant by one common sign, so the energies are equal; both sums run over the same
few thousand positive terms, 1e-11 relative bounds their rounding and that of H_II."""
import numpy as np
import pytest

from paper_2501_18185_gb300 import sci
from paper_2501_18185_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nroots", [1, 2, 3, 5, 8])
def test_far_from_reference(gpu, nroots):
    torch = gpu
    n, ne = 18, 9
    rng = np.random.default_rng(77)
    ints = W.real_integrals(rng, n, 2 * n, 0.9)
    low = (1 << ne) - 1
    strings = [low, low ^ (1 << 8) ^ (1 << 10), low ^ (1 << 3) ^ (1 << 12)]
    near = np.array(sorted(a | (b << n) for a in strings for b in strings), dtype=np.uint64)
    C = rng.normal(size=(len(near), nroots))
    C /= np.linalg.norm(C, axis=0)

    def back(key):
        return sum(1 << (n * (p // n) + n - 1 - p % n) for p in range(2 * n) if (int(key) >> p) & 1)

    far = np.array([back(k) for k in near], dtype=np.uint64)
    order = np.argsort(far)
    E0 = ints.h.trace() - 50.0 - np.arange(nroots)
    h, L = ints.h, ints.chol
    got = []
    for hh, LL, keys, c in ((h, L, near, C), (h[::-1, ::-1], L[:, ::-1, ::-1], far[order], C[order])):
        H = sci.Hamiltonian()
        H.set_integrals("spin_orbitals", np.ascontiguousarray(hh), chol=np.ascontiguousarray(LL))
        H.set_determinants(keys, ne, ne)
        got.append(H.enpt2(torch.from_numpy(np.ascontiguousarray(c)).cuda(), E0, table_bytes=1 << 26))
    assert got[0][3]["distinct_W"] == got[1][3]["distinct_W"]
    for x, y in zip(got[0][:3], got[1][:3]):
        assert np.allclose(x, y, rtol=1e-11, atol=0)
