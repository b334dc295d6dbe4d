"""The FP64 restriction, prolongation and node update over box sizes: one box
holding every node (its work lists span several staged chunks), boxes of odd
and unequal sizes, Z from the geometry and by value, with and without the
enriched modes.  One application of Algorithm 3 against the oracle's; the
tolerance is the preconditioner's (block condition numbers up to ~1e8 times
the FP64 round-off)."""
import numpy as np
import pytest
import torch

import xfem_inputs as X
from oracle import adef2 as O
from xfem_inputs import cracks as C

pytestmark = pytest.mark.gpu

# m hexes per axis, boxes per axis: 180 nodes in one box; 990 nodes (5 chunks of
# own nodes, 2 of coupled ones); 7^3 + 6^3-node boxes; a box with one layer
SIZES = [(5, 1), (9, 1), (13, 2), (7, 3)]


@pytest.mark.parametrize("m,n_box", SIZES)
@pytest.mark.parametrize("form", ["enriched", "rigid", "valued"])
def test_precond_box_sizes(m, n_box, form):
    from paper_2111_09294_gb300 import Solver
    P = X.build_problem(m, [C.PlanarEdgeCrack(0.5, 0.41, 1.25 / m)], n_box)
    K, M, Co = O.setup(P, enriched_modes=form != "rigid")
    kw = {}
    if form == "valued":
        Z, col0 = O.deflation_basis(P)
        Z = Z.tocsr()
        dof, sub = P.dof_ptr, P.sub_of_node
        kw = dict(z_cols=np.diff(col0).astype(np.int32), z_values=np.concatenate(
            [Z[dof[i]:dof[i + 1], col0[sub[i]]:col0[sub[i] + 1]].toarray().ravel()
             for i in range(P.n_nodes)]))
    s = Solver.from_problem(P, enriched_modes=form != "rigid", **kw)
    r = np.random.default_rng(m).standard_normal(P.n)
    z = s.precond(torch.tensor(r, device="cuda")).cpu().numpy()
    ref = O.adef2_apply(K, M, Co, r)
    assert np.linalg.norm(z - ref) <= 1e-8 * np.linalg.norm(ref)
    s.close()


# the FP32 iteration's row kernels: one unit per SM and many units (216 boxes),
# rows beyond the ones in flight before the wait (9, 1), coarse dimensions that
# are multiples of 4 and not.  tol 1e-12 and u to 1e-7 as for every mixed solve.
@pytest.mark.parametrize("m,n_box", SIZES + [(13, 6)])
def test_mixed_box_sizes(m, n_box):
    from paper_2111_09294_gb300 import Solver
    P = X.build_problem(m, [C.PlanarEdgeCrack(0.5, 0.41, 1.25 / m)], n_box)
    K, M, Co = O.setup(P)
    ref = O.adef2_pcg(K, P.f, M, Co, tol=1e-12)
    s = Solver.from_problem(P, precision="mixed")
    u, info = s.solve(torch.tensor(P.f, device="cuda"), tol=1e-12)
    assert info["rel_res_true"] <= 1e-12
    assert np.linalg.norm(u.cpu().numpy() - ref.u) <= 1e-7 * np.linalg.norm(ref.u)
    s.close()


# runs that end at every point of the host's look-ahead: the iteration cap at
# each of its first iterations, FP64 and mixed, streams and recorded graphs
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("graph", [False, True])
def test_iteration_caps(precision, graph):
    from paper_2111_09294_gb300 import Solver
    P = X.make("cube8_edge")
    f = torch.tensor(P.f, device="cuda")
    for cap in (0, 1, 2, 3, 4, 7, 8, 9, 17, 64):
        s = Solver.from_problem(P, precision=precision, graph=graph, max_iter=cap)
        _, info = s.solve(f, tol=1e-8, raise_on_error=False)
        done = info["rel_res_true"] <= 1e-8
        assert info["status"] == ("XDCG_OK" if done else "XDCG_NO_CONVERGENCE")
        assert done == (cap == 64) and (done or info["iterations"] == cap)
        s.close()
