"""Solves that fill the device: what one of them leaves with the context must not make the next one fail.

The device is filled by an allocation that leaves a stated number of bytes; the results are compared with those
of the same solve on an empty device."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
GB = 1 << 30


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _fill(torch, leave):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(int(free - leave), dtype=torch.uint8, device="cuda:0")


def _densities(s, sources):
    return s.observables()[0][sources]


def test_gmres_leaves_room_for_the_residual(torch_cuda, lib):
    """32 block columns of 8x8 sites and 100 points: 0.96 GB of state, 0.74 GB of slices for the residual and 0.21 GB
    a Krylov vector in 3.3 GB (and 0.3 that the first solve left).  The basis takes most of what is free when it is sized: the slices come first."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.uniform_problem("m", 8, 38, 24, 0.02, 1.0, 0.0, 0.05, 20.0, 1.0)
    sources = list(range(32))
    s = binding.Solver(p, device=0)
    s.build_sigma()
    s.solve(sources, precision=binding.PREC_F64, tol=1e-10)
    want = _densities(s, sources)
    s.close()
    s = binding.Solver(p, device=0)
    s.set_inner_solver(binding.INNER_GMRES)
    s.build_sigma()
    s.solve([0], precision=binding.PREC_TF32X3_F64REF, tol=1e-6)       # tables of Lambda
    hog = _fill(torch, int(3.3 * GB))
    try:
        res = s.solve(sources, precision=binding.PREC_TF32X3_F64REF, tol=1e-6)
        assert res.report["inner_gmres"] == 1 and res.report["chunks"] == 1
        assert np.abs(_densities(s, sources) - want).max() < 1e-5
    finally:
        del hog
        torch.cuda.empty_cache()
        s.close()


def test_chunks_do_not_depend_on_what_ran_before(torch_cuda, lib):
    """16 block columns of 8x8 sites and 128 points in 1.25 GB: the mixed solve keeps 0.67 GB of state and 0.34 GB of
    slices, the FP64 solve wants 0.54 and 0.54."""
    from paper_1309_5994_gb300 import binding
    torch = torch_cuda
    p = wl.uniform_problem("m", 8, 48, 32, 0.02, 1.0, 0.0, 0.05, 20.0, 1.0)
    sources = list(range(16))
    chunks, n = [], []
    for first_mixed in (False, True):
        s = binding.Solver(p, device=0)
        s.build_sigma()
        s.solve([0], precision=binding.PREC_TF32X3_F64REF, tol=1e-6)   # tables of Lambda
        s.solve([0], precision=binding.PREC_F64, tol=1e-10)
        hog = _fill(torch, int(1.25 * GB))
        try:
            if first_mixed:
                assert s.solve(sources, precision=binding.PREC_TF32X3_F64REF, tol=1e-6).report["chunks"] == 1
            for _ in range(2):
                chunks.append(s.solve(sources, precision=binding.PREC_F64, tol=1e-10).report["chunks"])
                n.append(_densities(s, sources))
        finally:
            del hog
            torch.cuda.empty_cache()
            s.close()
    assert chunks == [chunks[0]] * 4, chunks
    assert all(np.abs(x - n[0]).max() < 1e-9 for x in n)
