"""Sigma at the (N-2) bucket sizes where the double-excitation kernels meet: buckets of 2 to
4 members go through the register kernel, up to 64 through the sorted kernel or the aligned
walk, larger ones through the aligned walk.

One alpha and one beta electron share the empty (N-2) string, so a list of s such
determinants is one bucket of s members.  Every precision mode at one, two, three and eight
vectors equals the oracle (1e-11 relative; FP32 storage row by row within the rounding of
the pair table), over the whole list, over a row range and in the deterministic mode.
Spaces of three and four electrons mix the sizes in one table.
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
    rng = np.random.default_rng(700 + s)
    ints = W.real_integrals(rng, 14, 6, None)
    keys = np.sort(rng.choice(W.fci_keys(14, 1, 1), s, replace=False))
    return W.Workload(f"bucket_{s}", "spin_orbitals", 14, 1, 1, keys, ints, rng.normal(size=(s, 8)))


def _mixed(mode):
    if mode == "spinors":
        w = W.random_small(71, "spinors", 15, 4, 0, frac=0.25, nvec=4)
    else:
        w = W.random_small(73, "spin_orbitals", 9, 2, 2, frac=0.3, nvec=8)
    return w


SPACES = {f"bucket_{s}": (lambda s=s: _one_bucket(s)) for s in (2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 129)}
SPACES["mixed_real"] = lambda: _mixed("spin_orbitals")
SPACES["mixed_complex"] = lambda: _mixed("spinors")


def _check(S, C, o, prec):
    if prec == sci.SCI_PREC_F32_STORE_F64_ACC:
        rows = np.arange(len(C))
        A = o.sigma_abs_rows(rows, C)
        assert (np.abs(S - o.sigma_rows(rows, C).reshape(S.shape)) <= 1.05 * U32 * A.reshape(S.shape) + 1e-300).all()
    else:
        ref = o.sigma(C).reshape(S.shape)
        assert np.linalg.norm(S - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("name", list(SPACES))
def test_bucket_sizes(gpu, name):
    torch = gpu
    w = SPACES[name]()
    o = Oracle.from_workload(w)
    H = sci.Hamiltonian.from_workload(w)
    cplx = np.iscomplexobj(w.c)
    precs = [sci.SCI_PREC_F64, sci.SCI_PREC_F64_DS] + ([] if cplx else [sci.SCI_PREC_F32_STORE_F64_ACC])
    for prec in precs:
        for nvec in (1, 2, 3, 4) if cplx else (1, 2, 3, 8):
            C = np.ascontiguousarray(w.c[:, :nvec])
            t = torch.from_numpy(C).cuda()
            if prec == sci.SCI_PREC_F32_STORE_F64_ACC:
                t = t.float()
                C = t.double().cpu().numpy()
            S = H.sigma(t, prec=prec).cpu().numpy()
            _check(S, C, o, prec)
            a, b = w.M // 3, w.M - w.M // 4
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


def test_captured_and_repeated(gpu):
    """The chained launches of one sigma, captured in a CUDA graph and replayed on new
    coefficients, and back to back on one stream, where a launch that let its successor's
    successor start too early would mix two products."""
    torch = gpu
    w = W.selected_30o_cut(M=3000, seed=5)
    H = sci.Hamiltonian.from_workload(w)
    Cs = [torch.from_numpy(np.random.default_rng(k).normal(size=(w.M, 2))).cuda() for k in range(4)]
    ref = [H.sigma(C).cpu().numpy() for C in Cs]
    out = torch.empty((w.M, 2), dtype=torch.float64, device="cuda")
    for _ in range(20):
        got = []
        for C in Cs:
            H.sigma(C, out=out)
            got.append(out.clone())
        for r, g in zip(ref, got):
            assert np.abs(g.cpu().numpy() - r).max() <= 1e-13 * np.abs(r).max()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    H.set_stream(st)
    C = Cs[0].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        H.sigma(C, out=out)
    for k in (0, 1, 2, 3):
        C.copy_(Cs[k])
        graph.replay()
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - ref[k]).max() <= 1e-13 * np.abs(ref[k]).max()
