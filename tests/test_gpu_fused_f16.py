"""The fused sweep's FP16 operands: scales per row of Lambda W and per column group of X.

Hoppings that differ by orders of magnitude from bond to bond, and right-hand sides that do from column
group to column group, must not cost digits or overflow FP16."""
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


@pytest.mark.parametrize("variant", [2, 3])
@pytest.mark.parametrize("inner", [0, 1])
@pytest.mark.parametrize("jscale", [1e-6, 1.0, "mixed"])
def test_fused_solve_over_hopping_scales(torch_cuda, lib, jscale, inner, variant):
    """Refined to 1e-12 by the FP64-accurate residual; the number of refinements says what the FP32-accurate
    inner solves deliver (about three digits or more each)."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    Nc = 128 if variant == 2 else 256
    p = wl.small(L=3, Ly=2, Nt=3 * Nc // 8, Nm=Nc // 4, dt=0.02, beta=2.0, trap_c=0.3, U0=20.0)
    r = np.random.default_rng(11)
    f = jscale if jscale != "mixed" else 10.0 ** r.uniform(-6.0, 0.0, size=(p.Nb, 1))
    p = p.with_tables(J=p.J * f)
    S = dyson.setup(p)
    sources = [0, 4]
    ref = dyson.dense_solve(S, dyson.rhs_block_columns(S, sources))
    s = binding.Solver(p, device=0)
    s.set_sweep_variant(variant)
    s.set_inner_solver(inner)
    s.build_sigma()
    s.profile(True)
    g = torch.empty((len(sources), p.Nr, p.Nc, p.Nc), dtype=torch.complex128, device="cuda:0")
    res = s.solve(sources, precision=binding.PREC_TF32X3_F64REF, tol=1e-12, g_out=g)
    assert s.profile_query(binding.KERNEL_SWEEP_TC_FUSED)[0] > 0
    assert res.report["refinements"] <= 4
    got = g.cpu().numpy()
    for q in range(len(sources)):
        want = ref[:, :, q * p.Nc:(q + 1) * p.Nc]
        assert np.abs(got[q] - want).max() / np.abs(want).max() < 1e-11
    s.close()


@pytest.mark.parametrize("inner", [0, 1])
@pytest.mark.parametrize("Nt,Nm", [(9, 6), (12, 9), (24, 17), (38, 24), (48, 34), (70, 50), (72, 48), (96, 65), (120, 80)])
def test_fused_sweep_serves_every_contour(torch_cuda, lib, Nt, Nm, inner):
    """Contours that are no multiple of 64 (padded with zeros inside), of every tile form, with column counts and
    norm groups that end inside a 16-column chunk; no variant selected."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.random_tables(wl.small(L=3, Ly=2, Nt=Nt, Nm=Nm, dt=0.02, beta=1.0, trap_c=0.3, U0=14.0), seed=7, rel=0.1)
    S = dyson.setup(p)
    sources = [0, 4, 5]
    ref = dyson.dense_solve(S, dyson.rhs_block_columns(S, sources))
    s = binding.Solver(p, device=0)
    s.set_inner_solver(inner)
    s.build_sigma()
    s.profile(True)
    g = torch.empty((len(sources), p.Nr, p.Nc, p.Nc), dtype=torch.complex128, device="cuda:0")
    s.solve(sources, precision=binding.PREC_TF32X3_F64REF, tol=1e-12, g_out=g)
    assert s.profile_query(binding.KERNEL_SWEEP_TC)[0] > 0 and s.profile_query(binding.KERNEL_GATHER_TC)[0] == 0
    got = g.cpu().numpy()
    for q in range(len(sources)):
        want = ref[:, :, q * p.Nc:(q + 1) * p.Nc]
        assert np.abs(got[q] - want).max() / np.abs(want).max() < 1e-11
    sites, times = [k % p.Nr for k in range(40)], [(7 * k) % p.Nc for k in range(40)]
    v = torch.empty((40, p.Nr, p.Nc), dtype=torch.complex128, device="cuda:0")
    s.solve_vectors(sites, times, precision=binding.PREC_TF32X3_F64REF, tol=1e-12, g_out=v)
    want = dyson.dense_solve(S, dyson.rhs_vector_columns(S, list(zip(sites, times))))
    assert np.abs(v.cpu().numpy() - want.transpose(2, 0, 1)).max() / np.abs(want).max() < 1e-11
    s.close()


@pytest.mark.parametrize("Nt,Nm", [(7, 5), (8, 4), (200, 112)])
def test_gmres_item_shapes(torch_cuda, lib, Nt, Nm):
    """The GMRES vector kernels on strides they cannot load as float4 (19), on the CUDA-core stride (20) and on a
    contour of several items per column (512)."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.random_tables(wl.small(L=2, Ly=2, Nt=Nt, Nm=Nm, dt=0.01, beta=1.0, trap_c=0.3, U0=14.0), seed=9, rel=0.1)
    S = dyson.setup(p)
    ref = dyson.dense_solve(S, dyson.rhs_block_columns(S, [1, 2]))
    s = binding.Solver(p, device=0)
    s.set_inner_solver(1)
    s.build_sigma()
    g = torch.empty((2, p.Nr, p.Nc, p.Nc), dtype=torch.complex128, device="cuda:0")
    res = s.solve([1, 2], precision=binding.PREC_TF32X3_F64REF, tol=1e-12, g_out=g)
    assert res.report["inner_gmres"] == 1
    got = g.cpu().numpy()
    for q in range(2):
        want = ref[:, :, q * p.Nc:(q + 1) * p.Nc]
        assert np.abs(got[q] - want).max() / np.abs(want).max() < 1e-11
    s.close()


def test_gmres_states_that_start_at_eight_bytes(torch_cuda, lib):
    """Sites, columns and points all odd: the FP32 states of the CUDA-core stride start at a multiple of 8 bytes."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.random_tables(wl.small(L=3, Ly=1, Nt=10, Nm=1, dt=0.01, beta=0.2, trap_c=0.3, U0=14.0), seed=9, rel=0.1)
    S = dyson.setup(p)
    assert p.Nr * p.Nc % 2 == 1
    ref = dyson.dense_solve(S, dyson.rhs_block_columns(S, [1]))
    s = binding.Solver(p, device=0)
    s.set_inner_solver(1)
    s.build_sigma()
    g = torch.empty((1, p.Nr, p.Nc, p.Nc), dtype=torch.complex128, device="cuda:0")
    res = s.solve([1], precision=binding.PREC_TF32X3_F64REF, tol=1e-12, g_out=g)
    assert res.report["inner_gmres"] == 1
    assert np.abs(g.cpu().numpy()[0] - ref).max() / np.abs(ref).max() < 1e-11
    s.close()


@pytest.mark.parametrize("n,unfused", [(5440, False), (5472, True)])
def test_large_solves_of_64_points_take_the_unfused_form(torch_cuda, lib, n, unfused):
    """6 sites times n vector columns on either side of 32768, the rule's line at Nc = 64."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.random_tables(wl.small(L=3, Ly=2, Nt=24, Nm=16, dt=0.02, beta=1.0, trap_c=0.3, U0=14.0), seed=7, rel=0.1)
    S = dyson.setup(p)
    sites, times = [k % p.Nr for k in range(n)], [(7 * k) % p.Nc for k in range(n)]
    distinct = sorted(set(zip(sites, times)))
    ref = dict(zip(distinct, dyson.dense_solve(S, dyson.rhs_vector_columns(S, distinct)).transpose(2, 0, 1)))
    s = binding.Solver(p, device=0)
    s.build_sigma()
    s.profile(True)
    v = torch.empty((n, p.Nr, p.Nc), dtype=torch.complex128, device="cuda:0")
    s.solve_vectors(sites, times, precision=binding.PREC_TF32X3_F64REF, tol=1e-12, g_out=v)
    assert (s.profile_query(binding.KERNEL_GATHER_TC)[0] > 0) == unfused
    got, big = v.cpu().numpy(), max(np.abs(w).max() for w in ref.values())
    for k in list(range(0, n, 97)) + [n - 1]:
        assert np.abs(got[k] - ref[sites[k], times[k]]).max() / big < 1e-11
    s.close()


def _many_of_64(torch, binding, n, variant=None, leave=None):
    """profile counts (gather, single-CTA or default, fused) of a solve of n vector columns on 6 sites"""
    p = wl.random_tables(wl.small(L=3, Ly=2, Nt=24, Nm=16, dt=0.02, beta=1.0, trap_c=0.3, U0=14.0), seed=7, rel=0.1)
    s = binding.Solver(p, device=0)
    if variant is not None:
        s.set_sweep_variant(variant)
    s.build_sigma()
    hog = None
    if leave is not None:
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda:0")
    s.profile(True)
    res = s.solve_vectors([k % p.Nr for k in range(n)], [(7 * k) % p.Nc for k in range(n)],
                          precision=binding.PREC_TF32X3_F64REF, tol=1e-6)
    kinds = [s.profile_query(k)[0] for k in (binding.KERNEL_GATHER_TC, binding.KERNEL_SWEEP_TC, binding.KERNEL_SWEEP_TC_FUSED)]
    s.close()
    del hog
    torch.cuda.empty_cache()
    return kinds, res.report["chunks"]


@pytest.mark.parametrize("n,unfused", [(5440, False), (5472, True)])
def test_the_line_at_64_points_with_the_fused_form_selected(torch_cuda, lib, n, unfused):
    """As where none is selected: the fused form's tiles are half empty there."""
    from paper_1309_5994_gb300 import binding
    (gather, _, fused), _ = _many_of_64(torch_cuda, binding, n, variant=binding.SWEEP_FUSED_PAIR)
    assert (gather > 0) == unfused and (fused > 0) == (not unfused)


def test_the_line_at_64_points_counts_the_columns_of_a_chunk(torch_cuda, lib):
    """5472 columns of 6 sites in 96 MB are several chunks below the line."""
    from paper_1309_5994_gb300 import binding
    (gather, plain, _), chunks = _many_of_64(torch_cuda, binding, 5472, leave=96 << 20)
    assert chunks > 1 and gather == 0 and plain > 0


def test_the_tuned_form_is_the_one_that_runs(torch_cuda, lib):
    """Tuned on one block column of 6 sites (one launch a sweep beats two there), then used above the line."""
    from paper_1309_5994_gb300 import binding
    p = wl.random_tables(wl.small(L=3, Ly=2, Nt=24, Nm=16, dt=0.02, beta=1.0, trap_c=0.3, U0=14.0), seed=7, rel=0.1)
    s = binding.Solver(p, device=0)
    s.build_sigma()
    fused = binding.SWEEP_NAMES[s.autotune(1)["sweep_variant"]].startswith("fused")
    s.set_chunk(0)
    s.profile(True)
    n = 5472
    s.solve_vectors([k % p.Nr for k in range(n)], [(7 * k) % p.Nc for k in range(n)],
                    precision=binding.PREC_TF32X3_F64REF, tol=1e-6)
    assert (s.profile_query(binding.KERNEL_SWEEP_TC_FUSED)[0] > 0) == fused
    assert (s.profile_query(binding.KERNEL_GATHER_TC)[0] > 0) == (not fused)
    s.close()
