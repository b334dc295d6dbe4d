"""Contexts are independent: set-ups and solves of different contexts from
different host threads give what they give alone."""
import threading

import numpy as np
import pytest
import torch

import xfem_inputs as X
from xfem_inputs import cracks as C

pytestmark = pytest.mark.gpu


def _together(*jobs):
    """Runs the jobs in threads of their own, each on its own stream; their results."""
    out = [None] * len(jobs)

    def call(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            try:
                out[i] = jobs[i]()
            except Exception as e:      # an assertion of the caller shows it
                out[i] = e

    ts = [threading.Thread(target=call, args=(i,)) for i in range(len(jobs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return out


def test_setups_of_few_and_of_many_matrices_at_once():
    # one matrix to invert (E alone, many pivot steps) beside contexts with more
    # than sixteen caller blocks, over and over: the launches of the one must not
    # depend on what the other sets
    from paper_2111_09294_gb300 import Solver
    big = X.build_problem(18, [C.PlanarEdgeCrack(0.5, 0.41, 0.07)], 6)
    small = X.build_problem(5, [], 1)
    ptr = np.append(np.arange(0, small.n, 15), small.n)
    assert ptr.size - 1 > 16
    E = Solver.from_problem(big)
    r = torch.tensor(np.random.default_rng(2).standard_normal(big.n), device="cuda")
    ref = E.precond(r)
    stop = threading.Event()

    def one():
        try:
            for _ in range(80):
                s = Solver.from_problem(big)
                same = torch.equal(s.precond(r), ref)
                s.close()
                assert same
            return "same"
        finally:
            stop.set()

    def many():
        n = 0
        while not stop.is_set():
            Solver.from_problem(small, blocks=ptr).close()
            n += 1
        return n

    a, b = _together(one, many)
    assert a == "same", a
    assert isinstance(b, int) and b > 0, b
    E.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_solves_at_once_are_the_solves_alone(prec):
    # two host threads, a context, a stream and a load each: the same bits
    from paper_2111_09294_gb300 import Solver
    P = X.make("cube8_edge")
    F = [torch.tensor(f, device="cuda") for f in X.load_cases(P, 2, seed=3)]
    s = Solver.from_problem(P, precision=prec)
    ref = [s.solve(f) for f in F]
    s.close()

    def job(f, u, its):
        def run():
            s = Solver.from_problem(P, precision=prec)
            for _ in range(20):
                v, info = s.solve(f)
                assert info["iterations"] == its and torch.equal(u, v)
            s.close()
            return "same"
        return run

    torch.cuda.synchronize()
    out = _together(*[job(f, u, i["iterations"]) for f, (u, i) in zip(F, ref)])
    assert out == ["same", "same"], out
