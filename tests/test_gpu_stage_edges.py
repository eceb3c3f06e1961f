"""The 2D operator's stages at the edges of their rules, against the FP64 oracle: the row-walking forward
stage (rows_stream.cuh: row counts that end inside a chunk of 4 to 32 rows, widths at and below half the
length), the 16-points-per-thread columns (fft16.cuh: each length, problem counts that do and don't fill
a CTA's slots) and the stages of small complex128 batches (small64.cuh), each alone and inside a solve
whose scalar steps run in the last CTA of a launch (krylov_finish.cuh). The literal form's complex64
kernels (form_k.cu) likewise: each length, problem counts that do and don't fill a CTA's slots.

Tolerances: those of the other operator tests, 1e-5 (complex64: FP32 rounding 6e-8 times the depth of the
transforms and the stencil's cancellation) and 1e-10 (complex128) of A u, 20 times that of the
scattered part alone, and 1e-5 and 1e-8 for solutions."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2402_02116_gb300 import dbi, inputs
from paper_2402_02116_gb300.problem import DeviceProblem

pytestmark = pytest.mark.gpu

TOL = {dbi.C64: 1e-5, dbi.C128: 1e-10}


def oracle_for(w):
    return O.LSOracle(w.nz, w.nx, w.h, w.lz, w.lx, w.rho0, w.alpha0, w.beta0, w.omegas)


def check_apply(precision, nz, nx, n_src, freqs, literal=False, **lens):
    w = inputs.small_case(nz, nx, n_src=n_src, freqs=freqs, amp=0.15, **lens)
    P, orc, fs = DeviceProblem(w, precision), oracle_for(w), w.problem_fidx()
    u = inputs.seeded_complex((5, 2, nz, nx), nz + nx)
    pick = torch.arange(P.B, device=P.device) % 5
    out = (P.apply_k if literal else P.apply)(P.to_field(u)[pick].contiguous())
    apply = orc.apply_k if literal else orc.apply
    for b in sorted({0, P.B // 2, P.B - 2, P.B - 1} & set(range(P.B))):
        got, want = out[b].cpu().numpy(), apply(u[b % 5], w.model, fs[b])
        assert np.linalg.norm(got - want) < TOL[precision] * np.linalg.norm(want), b
        assert np.linalg.norm(got - want) < 20 * TOL[precision] * np.linalg.norm(want - u[b % 5]), b


# (nz, nx, n_src): FFT length 128 (33 to 64 columns), 256 and 512; the last has enough problems for chunks
# of 32 rows, the one before for 16
@pytest.mark.parametrize("nz, nx, n_src", [(5, 64, 1), (4, 33, 3), (13, 63, 2), (6, 128, 1), (35, 65, 2), (7, 256, 1),
                                           (34, 129, 2), (18, 131, 480), (40, 130, 960)])
def test_row_walking_stage(nz, nx, n_src):
    check_apply(dbi.C64, nz, nx, n_src, (9.0,))


# lengths 32 to 256, full and ragged
@pytest.mark.parametrize("nz", [9, 16, 17, 32, 33, 64, 65, 128])
@pytest.mark.parametrize("n_src", [1, 5, 16, 19])
def test_sixteen_point_columns(nz, n_src):
    check_apply(dbi.C64, nz, 7, n_src, (6.0, 11.0))


@pytest.mark.parametrize("nz, nx, lens", [(1, 3, {}), (8, 8, {}), (9, 8, {}), (8, 9, {}), (16, 16, {}), (17, 33, {}),
                                          (32, 64, {}), (33, 20, {}), (64, 64, {}), (64, 5, {}), (5, 64, {}),
                                          (7, 6, dict(lz=64, lx=128)), (9, 65, {}), (65, 9, {})])
@pytest.mark.parametrize("n_src", [1, 3])
def test_small_complex128_batches(nz, nx, lens, n_src):
    check_apply(dbi.C128, nz, nx, n_src, (6.0, 11.0), **lens)


@pytest.mark.parametrize("precision, nz, nx, n_src", [(dbi.C128, 9, 13, 1), (dbi.C128, 40, 64, 1), (dbi.C128, 12, 10, 2),
                                                      (dbi.C64, 9, 13, 1), (dbi.C64, 40, 33, 3), (dbi.C64, 12, 10, 160)])
def test_solves_match_oracle(precision, nz, nx, n_src):
    w = inputs.small_case(nz, nx, n_src=n_src, freqs=(7.0, 12.0))
    P, orc = DeviceProblem(w, precision), oracle_for(w)
    tol, bound = (1e-11, 1e-8) if precision == dbi.C128 else (1e-6, 1e-5)
    u, iters, relres, code = P.solve(P.incident(), tol=tol, max_iter=300, check_every=3)
    assert bool((code == dbi.CONVERGED).all())
    f, s = w.problem_fidx(), w.problem_src()
    for b in (0, P.B - 1):
        want = orc.solve(orc.incident(f[b], w.src_cells[s[b]], w.src_force[s[b]]), w.model, f[b], tol=1e-12)
        assert np.linalg.norm(u[b].cpu().numpy() - want) <= bound * np.linalg.norm(want), b


@pytest.mark.parametrize("nz, nx, lens", [(1, 3, {}), (9, 8, {}), (8, 9, {}), (17, 33, {}), (33, 65, {}), (64, 129, {}),
                                          (130, 20, {}), (5, 300, {}), (300, 5, {}), (7, 6, dict(lz=64, lx=512))])
@pytest.mark.parametrize("n_src", [1, 2, 9])
def test_literal_form_pairs(nz, nx, lens, n_src):
    check_apply(dbi.C64, nz, nx, n_src, (6.0, 11.0), literal=True, **lens)
