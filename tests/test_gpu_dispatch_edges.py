"""Calls on both sides of the rules that choose a kernel path, against the FP64 oracle: the length-512 columns of
complex64 (four problems per CTA or one, groups that straddle two frequencies, partial groups, compacted problem
lists), the tiles of complex128 batches (small ones where 256-thread tiles would leave much of their last wave
idle) and the kx slabs of 3D batches (the batch just large enough for the tables, the slab just small enough
for shared memory), with the products that reach the slabs without a stencil or with a perturbation as the model.

Tolerances: those of the other operator tests (test_gpu_stage_edges.py, test_gpu_3d.py)."""
import numpy as np
import pytest
import torch

from oracle import dbi_oracle3d as o3
from paper_2402_02116_gb300 import dbi, inputs
from paper_2402_02116_gb300.problem import DeviceProblem, DeviceProblem3D
from test_gpu_stage_edges import check_apply, oracle_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [129, 200, 256])
@pytest.mark.parametrize("n_src", [1, 5, 9, 19])  # of two frequencies: groups of one, 10, 18, 38 problems
def test_length_512_columns(nz, n_src):
    check_apply(dbi.C64, nz, 7, n_src, (6.0, 11.0))


def test_length_512_columns_of_a_compacted_batch():
    w = inputs.small_case(140, 9, n_src=9, freqs=(4.0, 12.0))
    P, orc = DeviceProblem(w, dbi.C64), oracle_for(w)
    rhs = P.incident()
    u, iters, _, code = P.solve(rhs, tol=1e-6, max_iter=300, check_every=1)
    assert bool((code == dbi.CONVERGED).all()) and int(iters.min()) > 0
    f, s = w.problem_fidx(), w.problem_src()
    for b in (0, 8, 9, P.B - 1):
        want = orc.solve(orc.incident(f[b], w.src_cells[s[b]], w.src_force[s[b]]), w.model, f[b], tol=1e-12)
        assert np.linalg.norm(u[b].cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want), b
    # all but five problems of both frequencies start at a solution: the launches run over a list of five
    left = [1, 7, 8, 10, 17]
    u0 = P.solve(rhs, tol=1e-7, max_iter=300)[0]
    u0[left] = 0
    again, iters2, _, code = P.solve(rhs, tol=1e-6, max_iter=300, check_every=1, u0=u0)
    assert bool((code == dbi.CONVERGED).all()) and [b for b in range(P.B) if iters2[b] > 0] == left
    assert torch.equal(iters2[left], iters[left])
    for b in left:
        assert torch.linalg.norm(again[b] - u[b]) <= 1e-5 * torch.linalg.norm(u[b]), b


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


def test_slab_products_match_oracle():
    w, P, orc = problem_3d(9, 11, 13, 12)
    assert P.B == 12
    U_b, _, _, code = P.solve(P.incident(), tol=1e-7, max_iter=500)
    assert bool((code == dbi.CONVERGED).all())
    rng = np.random.default_rng(5)
    dm = o3.reference_params_3d(w.rho0, w.alpha0, w.beta0)[:, None, None, None] * 0.01 * rng.standard_normal(
        (6, w.nz, w.ny, w.nx))
    r = P.to_field(rng.standard_normal((P.B, len(w.rec_cells), 3)) + 1j * rng.standard_normal((P.B, len(w.rec_cells), 3)))
    d, (_, _, cd) = P.frechet(U_b, P.to_model(dm), tol=1e-7)
    g, (_, _, cg) = P.adjoint(U_b, r, tol=1e-7)
    assert bool((cd == dbi.CONVERGED).all()) and bool((cg == dbi.CONVERGED).all())
    Ub, fidx = U_b.cpu().numpy().astype(np.complex128), list(w.problem_fidx())
    rec = [tuple(c) for c in w.rec_cells]
    want_d = o3.frechet_3d(orc, w.model, Ub, fidx, dm, rec, tol=1e-12)
    want_g = o3.adjoint_3d(orc, w.model, Ub, fidx, r.cpu().numpy().astype(np.complex128), rec, tol=1e-12)
    assert np.linalg.norm(d.cpu().numpy() - want_d) < 1e-4 * np.linalg.norm(want_d)
    assert np.linalg.norm(g.cpu().numpy() - want_g) < 1e-4 * np.linalg.norm(want_g)
