"""The split of the (N-2) table by bucket size, which sigma and the density matrices take their
bucket ranges from: a change of the tile threshold that fails half way changes nothing, and a
table out of size order is refused.  The library is linked here once more with allocations that
fail on request (the error code comes from the host, no GPU fault is involved).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2501_18185_gb300 import build, sci
from paper_2501_18185_gb300 import workloads as W

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(gpu, tmp_path_factory):
    out = tmp_path_factory.mktemp("split_probe")
    objs = [os.path.join(build.BUILD, s[:-3] + ".o") for s in build.SOURCES if s != "sci_setup.cu"]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    obj, lib = str(out / "split_probe.o"), str(out / "split_probe.so")
    for cmd in ([build.nvcc(), *build.NVCC_FLAGS, *build.ARCH, "-c", os.path.join(HERE, "split_probe.cu"), "-o", obj],
                [build.nvcc(), "-shared", "-Xlinker", "-Bsymbolic", *build.ARCH, obj, *objs, "-o", lib]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    return sci.load(lib)


@pytest.fixture
def space(probe, monkeypatch):
    monkeypatch.setattr(sci, "_lib", probe)
    w = W.random_small(73, "spin_orbitals", 9, 2, 2, frac=0.3, nvec=2)
    H = sci.Hamiltonian.from_workload(w)
    yield w, H
    probe.probe_limit_allocations(-1)
    H.close()


@pytest.mark.parametrize("ranged", [False, True])
def test_failed_threshold_changes_nothing(gpu, probe, space, ranged):
    torch = gpu
    w, H = space
    C = torch.from_numpy(w.c).cuda()
    a, b = (w.M // 3, w.M // 2) if ranged else (0, w.M)
    H.set_row_range(a, b)
    products = lambda: H.sigma(C).cpu().numpy()[a:b]  # noqa: E731
    S, (g1, g2) = products(), H.rdm12(C)
    assert np.abs(S).max() > 0
    for left in range(200):        # fails at the first, second, ... allocation of the call
        probe.probe_limit_allocations(left)
        rc = probe.sci_set_tile_threshold(H.ctx, 2)
        probe.probe_limit_allocations(-1)
        if rc == sci.SCI_OK:
            break
        assert np.abs(products() - S).max() <= 1e-13 * np.abs(S).max()
        assert torch.allclose(H.rdm12(C)[1], g2, rtol=0, atol=1e-13)
    assert left > 0 and rc == sci.SCI_OK
    assert np.abs(products() - S).max() <= 1e-13 * np.abs(S).max()


def test_table_out_of_order_is_refused(gpu, probe, space):
    _, H = space
    probe.probe_last_bucket_first.argtypes = [ctypes.c_void_p]
    assert probe.probe_last_bucket_first(H.ctx) == 0
    assert probe.sci_set_tile_threshold(H.ctx, 8) == sci.SCI_ERR_STATE
    assert "size order" in sci.sci_last_error(H.ctx)
