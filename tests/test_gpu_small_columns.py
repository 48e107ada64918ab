"""What a tolerance means: relative to every column of the right-hand side, and to the observables."""
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


@pytest.mark.parametrize("trap,below", [(30.0, 1e-12), (55.0, 1e-20), (105.0, 1e-40)])
def test_fp64_series_of_a_nearly_empty_site(torch_cuda, lib, trap, below):
    """The last contour point of a site high in the trap: every entry of the right-hand side carries the site's
    Boltzmann weight.  Same tolerance, relative to that column, as for any other."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.small(L=3, Ly=1, Nt=20, Nm=2, dt=0.05, beta=2.0, trap_c=trap, U0=4.0, J0=0.2)
    S = dyson.setup(p)
    site, time = 0, p.Nc - 1
    B = dyson.rhs_vector_columns(S, [(site, time)])
    scale = np.abs(B).max()
    assert 0.0 < scale < below
    want = dyson.dense_solve(S, B)[:, :, 0]
    s = binding.Solver(p, device=0)
    s.build_sigma()
    g = torch.empty((1, p.Nr, p.Nc), dtype=torch.complex128, device="cuda:0")
    res = s.solve_vectors([site], [time], precision=binding.PREC_F64, tol=1e-12, g_out=g)
    assert res.report["sweeps"] > 3
    assert np.abs(g.cpu().numpy()[0] - want).max() / scale < 1e-11
    s.close()


@pytest.mark.parametrize("Nt,Nm", [(48, 32), (38, 24), (96, 64)])
def test_loose_tolerance_with_a_short_time_step(torch_cuda, lib, Nt, Nm):
    """The double occupancy's difference quotient amplifies a residual by up to 2 / (dt U) = 500.  At a tolerance that the
    first refinement meets with little to spare, its error still stays within the tolerance."""
    from paper_1309_5994_gb300 import binding
    p = wl.random_tables(wl.small(L=3, Ly=2, Nt=Nt, Nm=Nm, dt=0.002, beta=1.0, trap_c=0.3, U0=2.0, J0=0.5), seed=4, rel=0.05)
    sources = list(range(p.Nr))
    s = binding.Solver(p, device=0)
    s.build_sigma()
    s.solve(sources, precision=binding.PREC_F64, tol=1e-13)
    want = s.observables()[2][:, 1:]
    first = s.solve(sources, precision=binding.PREC_TF32X3_F64REF, tol=1.0).report["residual"]
    tol = max(first / 0.18, 1.01e-8)
    res = s.solve(sources, precision=binding.PREC_TF32X3_F64REF, tol=tol)
    got = s.observables()[2][:, 1:]
    assert res.report["residual"] <= tol
    assert np.abs(got - want).max() < tol
    s.close()
