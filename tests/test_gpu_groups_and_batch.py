"""The FP64 product where its slice groups are launched as half blocks (the
matrix does not fill the SMs) and where they are not, and the batched kernels,
over sizes at which their work is divided differently."""
import numpy as np
import pytest
import torch

import xfem_inputs as X
from oracle import adef2 as O
from scipy.sparse.linalg import splu
from xfem_inputs import cracks as C

pytestmark = pytest.mark.gpu


# one group; a few; under and over 128 (one or more rounds of the last block's sum);
# close below and above the block slots of 152 SMs.  A row of t terms: both sums are
# within t / 2 eps |K||x| of the exact one; x^T y, summed in trees, adds less than
# its longest row: 512 eps |x|^T |K| |x|.
@pytest.mark.parametrize("m", [3, 6, 13, 22, 24, 32, 38])
def test_fp64_product_groups(m):
    from paper_2111_09294_gb300 import Solver
    P = X.build_problem(m, [C.PlanarEdgeCrack(0.5, 0.41, 1.25 / m)], max(1, m // 6))
    K = O.stiffness_csr(P)
    s = Solver.from_problem(P)
    x = np.random.default_rng(m).standard_normal(P.n)
    y, xty = s.spmv(torch.tensor(x, device="cuda"), "fp64")
    mag, eps = abs(K) @ abs(x), np.finfo(float).eps
    assert (abs(y.cpu().numpy() - K @ x) <= np.diff(K.indptr) * eps * mag).all()
    assert abs(float(xty) - x @ (K @ x)) <= 512 * eps * (abs(x) @ mag)
    s.close()


# columns padded to four and to eight; one unit per box and several; coarse
# dimensions that are multiples of four and not.  Residuals at tol 1e-10 and u to
# 1e-6, the condition number of these cubes being below 1e4 per scaled unknown.
@pytest.mark.parametrize("m,n_box", [(5, 1), (9, 1), (13, 2), (7, 3), (13, 6)])
@pytest.mark.parametrize("cols", [1, 3, 8])
def test_batch_box_sizes(m, n_box, cols):
    from paper_2111_09294_gb300 import Solver
    P = X.build_problem(m, [C.PlanarEdgeCrack(0.5, 0.41, 1.25 / m)], n_box)
    F = np.asarray(X.load_cases(P, cols, seed=m))
    s = Solver.from_problem(P, precision="mixed", max_batch=cols)
    U, infos = s.solve_batch(torch.tensor(F, device="cuda"), tol=1e-10)
    assert all(i["rel_res_true"] <= 1e-10 for i in infos)
    lu, U = splu(O.stiffness_csr(P).tocsc()), U.cpu().numpy()
    for j in range(cols):
        ref = lu.solve(F[j])
        assert np.linalg.norm(U[j] - ref) <= 1e-6 * np.linalg.norm(ref)
    s.close()
