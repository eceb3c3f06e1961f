"""A problem's solution does not depend on the batch it is solved in: alone, and as the first and the last of
a batch that shares the SMs among many problems, the complex64 BiCGSTAB gives the same bits and the same
iteration counts. (How a problem's sums are split into partials follows from the size of its grid; the batch only
sets how many CTAs work on them.) Grids on which a batch of 45 takes 1, 13, 13 and 16 CTAs per problem and a
problem alone 1, 32, 64 and 64, ragged ones among them."""
import pytest
import torch

from paper_2402_02116_gb300 import dbi, inputs
from paper_2402_02116_gb300.problem import DeviceProblem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz, nx", [(9, 13), (45, 180), (128, 128), (131, 250)])
def test_solution_alone_equals_solution_in_a_batch(nz, nx):
    w = inputs.small_case(nz, nx, n_src=1, freqs=(7.0,))
    one = DeviceProblem(w, dbi.C64)
    rhs = torch.cat([one.to_field(inputs.seeded_complex((1, 2, nz, nx), k)) for k in range(2)])

    def solve(fields):
        P = DeviceProblem(w, dbi.C64)
        P.fidx = torch.zeros(fields.shape[0], dtype=torch.int32, device=P.device)
        return P.solve(fields.contiguous(), tol=1e-6, max_iter=60, check_every=5)[:2]

    alone = [solve(rhs[k:k + 1]) for k in range(2)]
    u, iters = solve(rhs[torch.tensor([0] + [1] * 44, device=rhs.device)])
    for k, b in ((0, 0), (1, 1), (1, 44)):
        assert torch.equal(u[b], alone[k][0][0]) and iters[b] == alone[k][1][0], (k, b)
