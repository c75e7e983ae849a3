"""Recombination at the sizes where its kernels change path, against the oracle: lines of 1 to 15 nodes (in registers)
and longer ones (level by level), values on chip and in global memory (a line of 32,767 nodes), blocks of one node with
long lists of grids and blocks of more than 256 nodes.

Tolerance 1e-12: every result is a sum of surpluses over the levels of each axis (at most 15 + 1 of them) and over the
grids, whose coefficients' absolute sum stays below 2,000 on these sets: 2^-53 * 16 * 2000 = 4e-12 at worst, random
signs give well below 1e-12 in the 2-norm."""
import numpy as np
import pytest

import oracle
from paper_2509_22156_gb300 import binding as B
from paper_2509_22156_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_22156_gb300 import build
    build.build()
    B.load()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("d,n,L0", [(1, 1, 1), (1, 15, 1), (2, 10, 1), (2, 8, 3), (3, 7, 1), (4, 5, 1), (6, 4, 1)])
def test_recombination_matches_oracle(d, n, L0):
    P = B.Problem(d, n, L0, W.OP_HEAT)
    O = oracle.Problem(d, n, L0, W.OP_HEAT)
    u = W.random_vector(3 + d, P.n_total)
    ud = torch.from_numpy(u).cuda()
    out = torch.empty_like(ud)
    P.recombine(ud, out)
    ref = O.recombine(u)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    P.recombine(ud, ud)  # in place: the same kernels, the same sums
    assert torch.equal(ud, out)


def test_grids_in_global_memory_take_no_further_state():
    # the surpluses of every grid and of the sparse grid, and the plan; a grid too large for the chip is worked on in
    # the result's own place
    P = B.Problem(2, 17, 1, W.OP_HEAT)
    u = torch.from_numpy(W.random_vector(5, P.n_total)).cuda()
    out = torch.empty_like(u)
    n_sparse = 16 * 2 ** 17 + 1  # increments lam with |lam| <= n + 1: 2^(|lam| - 2) nodes each
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    P.recombine(u, out)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    assert taken <= 8 * (P.n_total + n_sparse) + (8 << 20)
    P.recombine(u, u)
    assert torch.equal(u, out)
