"""The complex64 3D operator with its y and z transforms fused per kx slab (csrc/ls3d_slab.cuh), against
the FP64 oracle. The path runs where a batch has about eight problems per frequency; these grids have
odd row counts, a half-empty last pair of depths, transform lengths at the edges of its range, and
batches that leave whole slots of its launches without a problem (converged ones, in the solve).

Tolerance: that of the other complex64 operator tests, 1e-5 of the scattered part (FP32 rounding 6e-8 times
the depth of three transforms each way and the stencil's cancellation)."""
import numpy as np
import pytest

from oracle import dbi_oracle3d as o3
from paper_2402_02116_gb300 import dbi, inputs

pytestmark = pytest.mark.gpu

# (nz, ny, nx): FFT lengths lz, ly, lx = fft_len of each
SHAPES = [(9, 11, 13), (5, 16, 33), (32, 9, 20), (33, 10, 12), (16, 64, 12), (8, 12, 128)]


def problem(shape, n_src=24, freqs=(9.0,)):
    from paper_2402_02116_gb300.problem import DeviceProblem3D
    w = inputs.small_case_3d(*shape, n_src=n_src, freqs=freqs, seed=sum(shape))
    return w, DeviceProblem3D(w, dbi.C64)


def oracle_for(w):
    return o3.LSOracle3D(w.nz, w.ny, w.nx, w.h, w.lz, w.ly, w.lx, w.rho0, w.alpha0, w.beta0, w.omegas)


@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_operator_matches_oracle(shape):
    w, P = problem(shape)
    u = inputs.seeded_complex((P.B, 3, *shape), 3)
    before = dbi.kernel_launches()
    got = P.apply(P.to_field(u)).cpu().numpy()
    # twiddles, the two scale kernels, tables, contrasts, stress, source + x, y-z, inverse x (the
    # separate passes: ten launches)
    assert dbi.kernel_launches() - before == 9, "the slab path did not run"
    orc, f = oracle_for(w), w.problem_fidx()
    for b in (0, P.B // 2, P.B - 1):
        want = orc.apply(u[b], w.model, f[b])
        assert np.linalg.norm(got[b] - want) <= 1e-5 * np.linalg.norm(want - u[b]), b


def test_solve_of_two_frequencies_matches_oracle():
    w, P = problem((9, 11, 13), n_src=25, freqs=(7.0, 12.0))
    u, iters, relres, code = P.solve(P.incident(), tol=1e-6, max_iter=200, check_every=4)
    assert bool((code == dbi.CONVERGED).all())
    u, orc, f, s = u.cpu().numpy(), oracle_for(w), w.problem_fidx(), w.problem_src()
    for b in (0, P.B - 1):
        want, _ = orc.solve(orc.incident(f[b], w.src_cells[s[b]], w.src_force[s[b]]), w.model, f[b], tol=1e-12)
        assert np.linalg.norm(u[b] - want) <= 1e-5 * np.linalg.norm(want), b
