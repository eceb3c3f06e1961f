"""Calls on both sides of the rules that choose a kernel path, against the FP64 oracle: the tiles of complex128
batches (small ones where 256-thread tiles would leave much of their last wave idle) and the kx slabs of 3D
batches (the batch just large enough for the tables, the slab just small enough for shared memory).

Tolerances: those of the other operator tests (test_gpu_stage_edges.py, test_gpu_3d.py)."""
import numpy as np
import pytest
import torch

from oracle import dbi_oracle3d as o3
from paper_2402_02116_gb300 import dbi, inputs
from paper_2402_02116_gb300.problem import DeviceProblem, DeviceProblem3D
from test_gpu_stage_edges import oracle_for

pytestmark = pytest.mark.gpu


# row tiles of 256 threads, and the tiles taken. Length 256: 76 small, 98 and 152 not, 154 small, 240 not; length 128:
# 64 and 112 small, 128 not; length 64: 303 small, 304 not. The columns take small ones at 64, 112, 196, 308
# and 480 tiles and not at 128, 152, 304, 606 and 608.
@pytest.mark.parametrize("nz, nx, B", [(16, 100, 38), (16, 100, 49), (16, 100, 76), (16, 100, 77), (16, 100, 120),
                                       (16, 50, 64), (16, 50, 112), (16, 50, 128), (32, 20, 303), (32, 20, 304)])
def test_complex128_tiles(nz, nx, B):
    w = inputs.small_case(nz, nx, n_src=1, freqs=(9.0,), amp=0.15)
    P, orc = DeviceProblem(w, dbi.C128), oracle_for(w)
    P.fidx = torch.zeros(B, dtype=torch.int32, device=P.device)
    u = inputs.seeded_complex((3, 2, nz, nx), nz + nx)
    field = P.to_field(u)[torch.arange(B, device=P.device) % 3].contiguous()
    out = P.apply(field)
    sol, _, _, code = P.solve(field, tol=1e-11, max_iter=200, check_every=3)
    assert bool((code == dbi.CONVERGED).all())
    for b in (0, B - 1):
        want = orc.apply(u[b % 3], w.model, 0)
        assert np.linalg.norm(out[b].cpu().numpy() - want) < 20e-10 * np.linalg.norm(want - u[b % 3]), b
        back = orc.apply(sol[b].cpu().numpy(), w.model, 0)
        assert np.linalg.norm(back - u[b % 3]) < 1e-9 * np.linalg.norm(u[b % 3]), b


def problem_3d(nz, ny, nx, n_src):
    w = inputs.small_case_3d(nz, ny, nx, n_src=n_src, freqs=(9.0,), seed=nz + ny + nx)
    P = DeviceProblem3D(w, dbi.C64)
    return w, P, o3.LSOracle3D(w.nz, w.ny, w.nx, w.h, w.lz, w.ly, w.lx, w.rho0, w.alpha0, w.beta0, w.omegas)


# (without slabs, with slabs): 11 | 12 problems; lz = 128 and ly = 64 with 62 | 60 depths; ly = 128 with 33 | 32
@pytest.mark.parametrize("outside, inside", [((9, 11, 13, 11), (9, 11, 13, 12)), ((62, 20, 12, 8), (60, 20, 12, 8)),
                                             ((33, 40, 12, 8), (32, 40, 12, 8))])
def test_slab_edges(outside, inside):
    counts = []
    for shape in (outside, inside):
        w, P, orc = problem_3d(*shape[:3], 1)
        P.fidx = torch.zeros(shape[3], dtype=torch.int32, device=P.device)
        u = inputs.seeded_complex((P.B, 3, *shape[:3]), 3)
        before = dbi.kernel_launches()
        got = P.apply(P.to_field(u))
        counts.append(dbi.kernel_launches() - before)
        for b in (0, P.B - 1):
            want = orc.apply(u[b], w.model, 0)
            assert np.linalg.norm(got[b].cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want - u[b]), (shape, b)
    assert counts[0] != counts[1]  # the two sides took different paths
