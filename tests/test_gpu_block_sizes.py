"""The FP32 product of the caller blocks' inverses (four rows and 128 columns at
a time, the first columns early) at block sizes below, at and above 96 and 128
and with rows that are no multiple of four times the warps.

Tolerances: the preconditioner is the oracle's up to FP32 rounding, and the
mixed solve ends at a replacement that waits for half the target, up to a third
of a decade more (40 iterations take eight): within a tenth plus two of the
oracle's iterations; u within 1e-6 at a residual of 1e-8 relative to f, by the
condition number below 1e2 of the preconditioned system."""
import numpy as np
import pytest
import torch

import xfem_inputs as X
from oracle import adef2 as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[3, 93, 96, 99, 126, 129, 132, 225], [33] * 30,
                                   [3] * 20 + [1500]])
def test_fp32_block_sizes(sizes):
    from paper_2111_09294_gb300 import Solver
    P = X.build_problem(9, [], 2)
    ptr = np.concatenate([[0], np.cumsum(sizes)])
    ptr = np.append(ptr, P.n) if ptr[-1] < P.n else ptr
    K, _, C = O.setup(P)
    M = O.SubdomainJacobi(K, [np.arange(a, b) for a, b in zip(ptr[:-1], ptr[1:])])
    its = O.adef2_pcg(K, P.f, M, C, tol=1e-8).iterations
    ref = O.adef2_pcg(K, P.f, M, C, tol=1e-12).u
    s = Solver.from_problem(P, precision="mixed", blocks=ptr)
    u, info = s.solve(torch.tensor(P.f, device="cuda"), tol=1e-8)
    assert info["n_fp64_iterations"] == 0 and info["rel_res_true"] <= 1e-8
    assert abs(info["iterations"] - its) <= 0.1 * its + 2
    assert np.linalg.norm(u.cpu().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)
    s.close()
