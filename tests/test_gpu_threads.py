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
