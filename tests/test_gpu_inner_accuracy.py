"""Accuracy of one FP32 inner solve on contours that are no multiple of 64.

The reference is the same series in full FP32: every product added with one rounding to nearest, in the order
of the contour (what the CUDA-core sweep does), in plain torch.  Both end on a rounding floor; its size is the
FP64 residual of the result."""
import math

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


def _fp32_series(torch, S, B, sweeps):
    """d after `sweeps` sweeps of d = r + Lambda W sum_j J d_j in FP32, each fused multiply-add rounded once (an
    FP32 product is exact in FP64; its sum is rounded to FP64, then to FP32)."""
    dev = "cuda:0"
    f32 = dict(dtype=torch.float32, device=dev)
    A = S.Lam * S.contour.W[None, None, :]
    Ar, Ai = (torch.tensor(np.ascontiguousarray(x), **f32) for x in (A.real, A.imag))
    J = torch.tensor(S.Jz, **f32)
    br, bi = (torch.tensor(np.ascontiguousarray(x), **f32) for x in (B.real, B.imag))
    fma = lambda c, a, b: (c.double() + a.double() * b.double()).float()
    dr, di = br.clone(), bi.clone()
    for _ in range(sweeps):
        xr, xi = torch.zeros_like(dr), torch.zeros_like(di)
        for i in range(S.Nr):
            for j, b in S.nbrs[i]:
                xr[i], xi[i] = fma(xr[i], J[b][:, None], dr[j]), fma(xi[i], J[b][:, None], di[j])
        yr, yi = torch.zeros_like(dr), torch.zeros_like(di)
        for k in range(S.Nc):
            lr, li, cr, ci = Ar[:, :, k, None], Ai[:, :, k, None], xr[:, None, k, :], xi[:, None, k, :]
            yr = fma(fma(yr, lr, cr), -li, ci)
            yi = fma(fma(yi, lr, ci), li, cr)
        dr, di = br + yr, bi + yi
    return (dr.double() + 1j * di.double()).cpu().numpy()


@pytest.mark.parametrize("Nc", [33, 50, 75, 100, 126, 139, 151, 170, 190, 195, 215, 250])
def test_inner_solve_is_as_accurate_as_full_fp32(torch_cuda, lib, Nc):
    """Geometric mean over three problems of residual / FP32 residual at most 1: the floors are sums of thousands of
    roundings whose ratio scatters by 20 % from problem to problem."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    ratios = []
    for k in range(3):
        Nm = max(4, Nc // (4 + 2 * (k % 2)))
        Nm -= (Nc - Nm) % 2
        p = wl.small(L=3, Ly=2, Nt=(Nc - Nm) // 2, Nm=Nm, dt=0.05, beta=1.0 if Nc < 60 else 2.0, trap_c=0.1, U0=20.0 - k)
        p = wl.random_tables(p, seed=k, rel=0.05)
        S = dyson.setup(p)
        n = 32
        cols = [(q % p.Nr, (7 * q + k) % p.Nc) for q in range(n)]
        B = dyson.rhs_vector_columns(S, cols)
        s = binding.Solver(p, device=0)
        s.set_inner_solver(binding.INNER_SERIES)
        s.build_sigma()
        res = s.solve_vectors([c[0] for c in cols], [c[1] for c in cols], precision=binding.PREC_TF32X3_F64REF, tol=1.0)
        assert res.report["refinements"] == 1
        d = _fp32_series(torch, S, B, res.report["sweeps"])
        r32 = np.abs(B - d + dyson.apply_K(S, d)).max() / np.abs(B).max()
        ratios.append(res.report["residual"] / r32)
        s.close()
    assert math.exp(np.mean(np.log(ratios))) <= 1.0, ratios
