"""A double build of more active orbitals than 48 KB of shared memory hold the diagonal of: J and K
against the same contractions by torch in double."""
import pytest

pytestmark = pytest.mark.gpu


def test_build_of_6160_active_orbitals():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as build
    build.build()
    import paper_2004_06142_gb300 as dn
    n, naux, npair = 6160, 3, 3080
    f64 = dict(dtype=torch.float64, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(0)
    B = torch.randn(naux, n, n, generator=g, **f64)
    B = (B + B.transpose(1, 2)).contiguous()
    C = torch.randn(n, n, generator=g, **f64) / n ** 0.5
    gamma = torch.rand(npair, generator=g, **f64)
    pair_map = torch.arange(npair, device="cuda").repeat(2).to(torch.int32)
    b = dn.Builder(n, naux, npair, 1, dn.PNOF7, dn.B_DENSE, dn.FP64)
    b.prepare(B)
    E, _, _ = b.forward(B[0].contiguous(), C, gamma, pair_map, want_lam=False)
    J, K = b.jk()
    assert b.status() == 0 and torch.isfinite(E).all()
    Jr, Kr = torch.zeros_like(J), torch.zeros_like(K)
    for P in range(naux):
        x = C.T @ (B[P] @ C)
        Jr += torch.outer(x.diagonal(), x.diagonal())
        Kr += x * x
    for a, r in ((J, Jr), (K, Kr)):
        # both round sums of n products of b twice over: far below 1e-12 of the largest
        assert (a - r).abs().max() <= 1e-12 * r.abs().max()
