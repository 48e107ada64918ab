"""The FP64 sweep and residual from BF16 slice products (k_oz64) against the oracle's dense solve.

Contour lengths at the edges of its tiles: shorter than one k-block, no multiple of 16, one point past a
row tile (2 Nc = 130), norm groups that end inside a warp's 16 columns (Nc = 40, 33), past one exact K
segment (2 Nc = 514, 600), and column counts that leave a remainder; hopping equal on every bond (J folded into the Lambda slices) and per bond."""
import numpy as np
import pytest

import workloads as wl
from oracle import dyson

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("Lx,Ly,Nt,Nm", [(1, 1, 2, 3), (2, 1, 1, 1), (3, 2, 8, 3), (4, 1, 16, 8),
                                         (2, 2, 15, 3), (2, 2, 24, 16), (3, 1, 25, 15), (2, 1, 96, 65), (2, 1, 120, 60)])
def test_fp64_sweep_and_residual_match_dense(torch_cuda, lib, Lx, Ly, Nt, Nm, uniform):
    """1e-12 of the largest entry, the FP64 path's tolerance (the slices keep 56 bits below each row's and
    column's largest value, so the sums are as exact as FP64 ones)."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.small(L=Lx, Ly=Ly, Nt=Nt, Nm=Nm, dt=0.02, beta=1.0, trap_c=0.3, U0=12.0, aU=0.1, aJ=0.2, omega=9.0)
    if not uniform:
        p = wl.random_tables(p, seed=3, rel=0.2)
    S = dyson.setup(p)
    sources = list(range(p.Nr))[:3]
    ref = dyson.dense_solve(S, dyson.rhs_block_columns(S, sources))
    s = binding.Solver(p, device=0)
    s.build_sigma()
    for prec, kind in ((binding.PREC_F64, binding.KERNEL_SWEEP_F64), (binding.PREC_TF32X3_F64REF, None)):
        g = torch.empty((len(sources), p.Nr, p.Nc, p.Nc), dtype=torch.complex128, device="cuda:0")
        s.profile(True)
        res = s.solve(sources, precision=prec, tol=1e-13, g_out=g)
        if kind is not None:
            assert s.profile_query(kind)[0] == res.report["sweeps"]
        got = g.cpu().numpy()
        for q in range(len(sources)):
            want = ref[:, :, q * p.Nc:(q + 1) * p.Nc]
            assert np.abs(got[q] - want).max() / np.abs(want).max() < 1e-12, prec
    s.close()


def test_vector_columns_leave_a_column_remainder(torch_cuda, lib):
    """33 vector columns (two norm groups of 32, the second padded): one 64-column tile."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.random_tables(wl.small(L=3, Ly=2, Nt=10, Nm=7, trap_c=0.2, U0=10.0), seed=5, rel=0.1)
    S = dyson.setup(p)
    sites = [k % p.Nr for k in range(33)]
    times = [(5 * k) % p.Nc for k in range(33)]
    ref = dyson.dense_solve(S, dyson.rhs_vector_columns(S, list(zip(sites, times))))
    s = binding.Solver(p, device=0)
    s.build_sigma()
    g = torch.empty((33, p.Nr, p.Nc), dtype=torch.complex128, device="cuda:0")
    s.solve_vectors(sites, times, precision=binding.PREC_F64, tol=1e-13, g_out=g)
    got = g.cpu().numpy()
    for k in range(33):
        assert np.abs(got[k] - ref[:, :, k]).max() / np.abs(ref).max() < 1e-12
    s.close()


def test_expired_wait_of_the_fp64_sweep_returns_timeout(torch_cuda, lib):
    from paper_1309_5994_gb300 import binding
    p = wl.small(L=3, Ly=3, Nt=40, Nm=20, trap_c=0.3, U0=20.0)
    s = binding.Solver(p, device=0)
    s.build_sigma()
    try:
        s.set_wait_limit(1e-9)
        with pytest.raises(binding.DysonError) as e:
            s.solve([0, 3], precision=binding.PREC_F64, tol=1e-12)
        assert e.value.code == -5
    finally:
        s.set_wait_limit(0.0)
    assert s.solve([0, 3], precision=binding.PREC_F64, tol=1e-12).status == 0
    s.close()
