"""donof_prepare_B (mixed precision) at the sizes where its passes over the slices change their
shared memory: every size that donof_workspace_size accepts is converted, and packed slices give
the builds of dense ones, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()


def _slices(nbf, naux):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nbf)
    B = torch.randn(naux, nbf, nbf, dtype=torch.float64, device="cuda", generator=g)
    for P in range(naux):
        B[P] += B[P].T.clone()
    return B


def _agree(nbf, naux):
    import torch
    import paper_2004_06142_gb300 as dn
    dense = _slices(nbf, naux)
    g = torch.Generator(device="cuda").manual_seed(naux)
    C = torch.randn(nbf, nbf, dtype=torch.float64, device="cuda", generator=g) / nbf ** 0.5
    h = dense[0] / 8
    gamma = torch.tensor([0.3, 0.9], dtype=torch.float64, device="cuda")
    pair_map = torch.tensor([0, 1, 0, 1], dtype=torch.int32, device="cuda")
    mu, nu = torch.tril_indices(nbf, nbf, device="cuda")
    out = []
    for layout, B in ((dn.B_DENSE, dense), (dn.B_PACKED, dense[:, mu, nu].contiguous())):
        b = dn.Builder(nbf, naux, 2, 1, dn.PNOF7, layout, dn.MIXED)
        b.prepare(B)
        out.append(b.forward(h, C, gamma, pair_map) + b.backward(torch.ones_like(gamma[:1])))
        torch.cuda.synchronize()
        assert b.status() == 0
    for x, y in zip(*out):
        assert torch.isfinite(x).all() and torch.equal(x, y)


# dynamic shared memory just below 48 KB: packed slices' sums, dense slices' scale exponents
@pytest.mark.parametrize("nbf", [338, 339, 340, 341, 342])
def test_packed_at_the_default_limit(nbf):
    _agree(nbf, 60)


@pytest.mark.parametrize("nbf", [12032, 12200, 12288])
def test_dense_at_the_default_limit(nbf):
    import torch
    import paper_2004_06142_gb300 as dn
    b = dn.Builder(nbf, 80, 2, 1, dn.PNOF7, dn.B_DENSE, dn.MIXED)
    b.prepare(torch.ones(80, nbf, nbf, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    assert b.status() == 0


# the largest packed slices whose column sums get two warps' shares of shared memory, and whole rows
# gathered beyond, each with slices enough for a CTA each and with few
@pytest.mark.parametrize("nbf,naux", [(4266, 192), (4267, 130), (4267, 3), (6400, 1), (6401, 2)])
def test_packed_beyond_shared_memory(nbf, naux):
    _agree(nbf, naux)


# the fewest slices that get a CTA each (80 dense, 384 / 8 packed) and the most that do not
@pytest.mark.parametrize("nbf", [4, 9, 130, 257, 301])
@pytest.mark.parametrize("naux", [1, 47, 48, 79, 80])
def test_few_slices(nbf, naux):
    _agree(nbf, naux)


@pytest.mark.parametrize("naux", [1, 130])
def test_packed_beyond_shared_memory_reports_non_finite(naux):
    import torch
    import paper_2004_06142_gb300 as dn
    for bad in (float("inf"), float("nan")):
        b = dn.Builder(4300, naux, 2, 1, dn.PNOF7, dn.B_PACKED, dn.MIXED)
        B = torch.ones(naux, 4300 * 4301 // 2, dtype=torch.float64, device="cuda")
        B[naux - 1, 4299 * 4300 // 2 + 17] = bad  # in the last row: part of column 17 too
        b.prepare(B)
        torch.cuda.synchronize()
        assert b.status() == -3
