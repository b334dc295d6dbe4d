"""The blocked FP64 inverse at the edges of its 64 x 64 tiles: caller blocks of
sizes around multiples of 64 (several matrices of different tile counts in one
batch, the last pivot block partly filled) and one large block (27 steps),
through one application of Algorithm 3 against dense solves.  Tolerance: the
preconditioner's 1e-8 (explicit inverses, condition numbers up to ~1e5 here)."""
import numpy as np
import pytest
import torch

import xfem_inputs as X
from oracle import adef2 as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[3, 63, 66, 126, 129, 189, 192, 195, 258], [66] * 20, [1923]])
def test_block_inverse_sizes(sizes):
    from paper_2111_09294_gb300 import Solver
    P = X.build_problem(9, [], 2)
    ptr = np.concatenate([[0], np.cumsum(sizes)])
    ptr = np.append(ptr, P.n) if ptr[-1] < P.n else ptr
    K, _, C = O.setup(P)
    M = O.SubdomainJacobi(K, [np.arange(a, b) for a, b in zip(ptr[:-1], ptr[1:])])
    s = Solver.from_problem(P, blocks=ptr)
    r = np.random.default_rng(1).standard_normal(P.n)
    z = s.precond(torch.tensor(r, device="cuda")).cpu().numpy()
    ref = O.adef2_apply(K, M, C, r)
    assert np.linalg.norm(z - ref) <= 1e-8 * np.linalg.norm(ref)
    s.close()
