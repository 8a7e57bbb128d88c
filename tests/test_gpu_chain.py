"""Chained launches of a build and the buffers it clears on the way (csrc/common.cuh): a build on
a used workspace, behind kernels that still write its inputs, and replayed as a graph gives the
bits of a fresh one.  Nothing in a build depends on scheduling, so the results are compared bit
for bit.  Sizes: grids all chained; J, K and Y wider than the chained ones; K = 640 and 641, the
last double build whose first kernel clears the buffers and the first that uses memsets; blocks of
slices; a contraction that fills the chip."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MIXED, FP64 = "mixed", "fp64"


@pytest.fixture(scope="module")
def dn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()
    import paper_2004_06142_gb300 as dn
    return dn


@pytest.mark.parametrize("nbf,naux,npair,ncwo,precision,budget", [
    (24, 96, 5, 1, MIXED, 0), (24, 96, 5, 1, FP64, 0), (33, 70, 4, 2, FP64, 1 << 18),
    (33, 70, 4, 2, MIXED, 1 << 18), (120, 480, 8, 4, MIXED, 0), (200, 900, 20, 3, MIXED, 0),
    (200, 900, 20, 3, FP64, 0), (640, 40, 4, 2, FP64, 0), (641, 40, 4, 2, FP64, 0)])
def test_reused_behind_writers_and_replayed(dn, nbf, naux, npair, ncwo, precision, budget):
    import torch
    A = npair * (1 + ncwo)
    g = torch.Generator(device="cuda")
    g.manual_seed(nbf + naux)

    def rand(*shape):
        return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)

    B = rand(naux, nbf, nbf) - 0.5
    B = (B + B.transpose(1, 2)) / naux ** 0.5
    h = rand(nbf, nbf) - 0.5
    h = h + h.T
    pm = torch.tensor(list(range(npair)) + [i // ncwo for i in range(npair * ncwo)],
                      dtype=torch.int32, device="cuda")
    sets = [(torch.linalg.qr(rand(nbf, nbf))[0].contiguous(), rand(npair * ncwo)) for _ in range(2)]
    one = torch.ones(1, dtype=torch.float64, device="cuda")

    def builder():
        bld = dn.Builder(nbf, naux, npair, ncwo,
                         precision=dn.MIXED if precision == MIXED else dn.FP64,
                         x_budget_bytes=budget)
        bld.prepare(B)
        return bld

    def run(bld, C, gamma):
        E, lam, dEdg = bld.forward(h, C, gamma, pm)
        return (E, lam, dEdg) + tuple(bld.backward(one))

    want = [[t.cpu().numpy() for t in run(builder(), C, gm)] for C, gm in sets]
    assert all(np.isfinite(t).all() for w in want for t in w)
    for lam in (w[1] for w in want):  # cleared beyond the active columns
        assert (lam[:, A:] == 0).all() and (lam[:, :A] != 0).any()

    used = builder()
    C, gm = torch.zeros_like(sets[0][0]), torch.zeros_like(sets[0][1])
    run(used, *sets[1])
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for k in (0, 1, 0):
            for _ in range(20):  # the inputs are still being written when the build is queued
                C.copy_(sets[1 - k][0])
                gm.copy_(sets[1 - k][1])
            C.copy_(sets[k][0])
            gm.copy_(sets[k][1])
            # outputs' memory holds NaN
            junk = [torch.full((nbf, nbf), np.nan, dtype=torch.float64, device="cuda")
                    for _ in range(4)]
            del junk
            out = run(used, C, gm)
            stream.synchronize()
            for w, o in zip(want[k], out):
                np.testing.assert_array_equal(w, o.cpu().numpy())
    torch.cuda.synchronize()

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = run(used, C, gm)
    for k in (1, 0):
        C.copy_(sets[k][0])
        gm.copy_(sets[k][1])
        for o in out:
            o.fill_(np.nan)
        graph.replay()
        torch.cuda.synchronize()
        for w, o in zip(want[k], out):
            np.testing.assert_array_equal(w, o.cpu().numpy())
