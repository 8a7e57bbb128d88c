"""donof_workspace_size works out the blocks of slices that every call works out again: its host
time stays small whatever the number of blocks."""
import time

import pytest


@pytest.fixture(scope="module")
def dn():
    import paper_2004_06142_gb300.build as b
    b.build()
    import paper_2004_06142_gb300 as dn
    return dn


@pytest.mark.parametrize("nbf,naux,budget", [(24, 1_000_000, 16000), (24, 16_000_000, 10000),
                                             (200, 60_000, 40_000), (24, 96, 0)])
def test_many_blocks_cost_little_host_time(dn, nbf, naux, budget):
    from paper_2004_06142_gb300 import binding as bd
    prob = bd.make_problem(nbf, naux, 5, 1, x_budget_bytes=budget)
    t = time.perf_counter()
    for _ in range(100):
        assert bd.donof_workspace_size(prob) > 0
    # about a millisecond; a layout for every number of blocks took 0.1 to 2 s
    assert time.perf_counter() - t < 0.05
