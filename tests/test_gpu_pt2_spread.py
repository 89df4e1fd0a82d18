"""ENPT2 with integrals of very different sizes: one orbital is shifted far up (a penalty that
keeps it out of the space), so the one-electron terms of H_II span 2^36, while the determinants
that matter leave it empty.  Their H_II are as accurate as without the shift: both the device and
the oracle form them in FP64 sums of some hundred terms, whose rounding of about 1e-14 stands
against denominators of order one; with up to 1e5 terms of E2 in different order, 1e-10 relative
as in the other comparisons with the oracle.  A shift beyond the FP64 range gives no number.
"""
import numpy as np
import pytest

from oracle import Oracle
from oracle import pt2 as PT
from paper_2501_18185_gb300 import sci
from paper_2501_18185_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _space(mode, n, na, nb, nroots):
    """A random space without the highest orbital, its lowest roots, and the shifted orbitals."""
    w = W.random_small(311, mode, n, na, nb, naux=6, frac=0.4)
    high = [n - 1] if mode == "spinors" else [n - 1, 2 * n - 1]
    w.keys = w.keys[~np.any([(w.keys >> np.uint64(p)) & np.uint64(1) == 1 for p in high], axis=0)]
    ev, U = np.linalg.eigh(Oracle.from_workload(w).dense())
    return w, U[:, :nroots].copy(), ev[:nroots].copy()


@pytest.mark.parametrize("mode,n,na,nb", [("spin_orbitals", 8, 3, 3), ("spinors", 11, 4, 0)])
@pytest.mark.parametrize("nroots", [1, 3])
@pytest.mark.parametrize("shift", [0.0, 2.0 ** 12, 2.0 ** 36])
def test_shifted_orbital(gpu, mode, n, na, nb, nroots, shift):
    torch = gpu
    w, C, E0 = _space(mode, n, na, nb, nroots)
    w.ints.h[n - 1, n - 1] += shift
    ref = PT.enpt2(mode, n, na, w.n_beta, w.ints.h, w.ints.eri(), w.keys, C, E0)
    H = sci.Hamiltonian.from_workload(w)
    e2q = H.enpt2(torch.from_numpy(C).cuda(), E0)[2]
    assert np.abs(ref).min() > 1e-3
    assert np.allclose(e2q, ref, rtol=1e-10, atol=0), (e2q, ref)


def test_sums_beyond_fp64_are_no_number(gpu):
    torch = gpu
    w, C, E0 = _space("spin_orbitals", 6, 2, 2, 1)
    w.ints.h[5, 5] = 1.7e308
    H = sci.Hamiltonian.from_workload(w)
    e2q = H.enpt2(torch.from_numpy(C).cuda(), E0)[2]
    assert not np.isfinite(e2q).any()
