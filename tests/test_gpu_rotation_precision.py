"""What the rotation leaves, measured on fp32 inputs against 64-bit products. A row takes part in about 1e4 rotations; each
may round to nearest (2^-24 of the row's length, either way), so the lengths of the rows, and with them the diagonal of
U^T U - I, may drift like the square root of that number: 2^-24 * 1e2 = 6e-6. In proportion to it, as a bias of the rotations
adds up, would be 6e-4."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def planted(seed, L, d, k, decades):
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.linalg.qr(torch.randn((L, k), generator=g, device="cuda", dtype=torch.float64))[0]
    v = torch.linalg.qr(torch.randn((d, k), generator=g, device="cuda", dtype=torch.float64))[0]
    s = 10.0 ** (-decades * torch.arange(k, device="cuda", dtype=torch.float64) / (k - 1))
    return ((u * (s / s.norm())) @ v.T * (L * d) ** 0.5).float()


# with the roots of the rotation uncorrected 9.4e-5 / 4.7e-5 / 6.1e-5, with one Newton step 3.6e-6 / 2.0e-6 / 3.2e-6
@pytest.mark.parametrize("L,d,r", [(1024, 2048, 960), (2048, 512, 400), (1024, 1024, 512)])
def test_row_lengths_do_not_drift(L, d, r):
    import paper_2403_02352_b200 as atp
    c = atp.Context(0)
    try:
        U, _, _ = atp.atp_principal_basis(c, planted(0, L, d, min(L, d), 6), [L], [r])
        c.poll()
        u = U.double()
        assert (u.T @ u - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max().item() <= 1e-5
    finally:
        c.close()
