"""dyson_set_slice_memory: the FP64-pipe kernels where slices may not be made, and the adjoint's site contraction on
the tensor cores against the FP64-pipe one."""
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
@pytest.mark.parametrize("Lx,Ly,Nt,Nm", [(1, 1, 2, 3), (3, 2, 8, 3), (4, 1, 16, 8), (2, 2, 15, 3), (2, 2, 24, 16), (2, 1, 96, 65)])
def test_fp64_pipe_sweep_and_residual_match_dense(torch_cuda, lib, Lx, Ly, Nt, Nm, uniform):
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.small(L=Lx, Ly=Ly, Nt=Nt, Nm=Nm, dt=0.02, beta=1.0, trap_c=0.3, U0=12.0, aU=0.1, aJ=0.2, omega=9.0)
    if not uniform:
        p = wl.random_tables(p, seed=3, rel=0.2)
    S = dyson.setup(p)
    sources = list(range(p.Nr))[:3]
    ref = dyson.dense_solve(S, dyson.rhs_block_columns(S, sources))
    s = binding.Solver(p, device=0)
    s.set_slice_memory(0)
    s.build_sigma()
    for prec in (binding.PREC_F64, binding.PREC_TF32X3_F64REF):
        g = torch.empty((len(sources), p.Nr, p.Nc, p.Nc), dtype=torch.complex128, device="cuda:0")
        s.profile(True)
        res = s.solve(sources, precision=prec, tol=1e-13, g_out=g)
        if prec == binding.PREC_F64:
            assert s.profile_query(binding.KERNEL_SWEEP_F64)[0] == res.report["sweeps"]
        else:
            assert s.profile_query(binding.KERNEL_RESIDUAL_F64)[0] == res.report["refinements"]
            assert s.profile_query(binding.KERNEL_RESIDUAL_SPLIT)[0] == 0
        got = g.cpu().numpy()
        for q in range(len(sources)):
            want = ref[:, :, q * p.Nc:(q + 1) * p.Nc]
            assert np.abs(got[q] - want).max() / np.abs(want).max() < 1e-12, prec
    with pytest.raises(binding.DysonError):
        s.set_slice_memory(-2)
    s.close()


# 8 Nr^2 Nc^2 above 1e9, from which the contraction runs on the tensor cores; rows 2 Nc below, above and at no
# multiple of a tile of 128, columns Nc at no multiple of 64, sums 2 Nr of one exact segment of 512 and of several
# with a remainder
@pytest.mark.parametrize("Lx,Ly,Nt,Nm", [(20, 19, 12, 9), (14, 13, 36, 28), (25, 24, 8, 3), (9, 9, 60, 27)])
def test_site_contraction_on_the_tensor_cores(torch_cuda, lib, Lx, Ly, Nt, Nm):
    """Two sites at a time in slices against the FP64 pipe, on the same solves (neither context may keep slices of
    Lambda): the products keep 2^-56 of the largest entry each, so the gradients agree to FP64 rounding."""
    from paper_1309_5994_gb300 import binding
    p = wl.random_tables(wl.uniform_problem("c", Lx, Nt, Nm, 0.05, 1.0, 0.0, 0.01, 18.0, 1.0, Ly=Ly), seed=2, rel=0.05)
    assert 8.0 * p.Nr ** 2 * p.Nc ** 2 > 1e9
    r = np.random.default_rng(1)
    wn, wd = r.uniform(0.0, 1.0, p.Nr), r.uniform(0.0, 1.0, p.Nr)
    per_site = 8 * 2 * p.Nc * (-(-2 * p.Nr // 32) * 32) * 2 * 3 // 2 + 12 * p.Nc
    grads = []
    for memory in (0, 2 * per_site + 1000, -1):
        s = binding.Solver(p, device=0)
        s.set_slice_memory(memory)
        s.build_sigma()
        before = s.launch_count()
        _, gU, gJ, res = s.adjoint_obs(wn, wd, precision=binding.PREC_F64, tol=1e-13)
        grads.append((gU, gJ, s.launch_count() - before))
        s.close()
    (u0, j0, _), (u1, j1, n1), (u2, j2, n2) = grads
    assert n1 > 3 * (p.Nr // 2)                                           # two sites at a time
    assert np.abs(j1 - j0).max() < 1e-14 * np.abs(j0).max()               # (does not involve the contraction)
    assert np.abs(u1 - u0).max() < 1e-13 * np.abs(u0).max()
    assert np.abs(u2 - u0).max() < 1e-12 * np.abs(u0).max() and np.abs(j2 - j0).max() < 1e-12 * np.abs(j0).max()
