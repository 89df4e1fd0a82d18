"""The expansion of the density matrices at orbital counts around a warp of 32 and below one, real
and complex, against the oracle (1e-12 absolute for normalised vectors, as in the other tests of
these calls: sums of at most a few hundred products below one).  The buffers handed in hold
numbers before, and every element of them is written."""
import numpy as np
import pytest

from oracle import Oracle
from paper_2501_18185_gb300 import sci
from paper_2501_18185_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,n,na,nb", [("spinors", 3, 2, 0), ("spinors", 31, 3, 0), ("spinors", 32, 3, 0),
                                          ("spinors", 33, 3, 0), ("spin_orbitals", 1, 1, 1), ("spin_orbitals", 2, 1, 2),
                                          ("spin_orbitals", 16, 2, 1), ("spin_orbitals", 17, 1, 2)])
def test_every_element(gpu, mode, n, na, nb):
    torch = gpu
    w = W.random_small(400 + n, mode, n, na, nb, frac=0.08 if n > 8 else 1.0)
    H = sci.Hamiltonian.from_workload(w)
    C = torch.from_numpy(w.c).cuda()
    no = H.norb
    g1 = torch.full((no, no), 7.0, dtype=C.dtype, device="cuda")
    g2 = torch.full((no, no, no, no), 7.0, dtype=C.dtype, device="cuda")
    sci.sci_rdm12(H.ctx, C, 1, None, g1, g2)
    r1, r2 = Oracle.from_workload(w).rdm12(np.ascontiguousarray(w.c[:, 0]))
    assert np.abs(g1.cpu().numpy() - r1).max() < 1e-12
    assert np.abs(g2.cpu().numpy() - r2).max() < 1e-12
    only1 = H.rdm12(C, rdm2=False)[0]
    assert (only1 - g1).abs().max() < 1e-12
