"""How the CTAs of the rotation and of the orthonormalisation are dealt out: batches that fill an SM once, that keep the second
CTA of the pivots' SMs away, that use every CTA, and that have more pairs of blocks than SMs; iterates whose Gram matrix goes by
half tiles, partly filled ones among them, and by whole tiles. Bounds: those of the parity tests (orthogonality to the storage
type's rounding, X_r against U^T X to 8 roundings, scaled off-diagonals to the rotation's threshold)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def states(seed, lengths, d, planted, dtype):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for L in lengths:
        k = min(planted, L, d)
        u = torch.linalg.qr(torch.randn((L, k), generator=gen, device="cuda"))[0]
        v = torch.linalg.qr(torch.randn((d, k), generator=gen, device="cuda"))[0]
        s = 10.0 ** (-1.5 * torch.arange(k, device="cuda") / k) * (L * d / k) ** 0.5
        out.append((u * s) @ v.T + 0.02 * torch.randn((L, d), generator=gen, device="cuda"))
    return torch.cat(out).to(dtype)


@pytest.mark.parametrize("lengths,d,r,dtype", [
    ([512], 512, 120, torch.float32),                  # a few CTAs, one to an SM
    ([1500], 1600, 1000, torch.bfloat16),              # 17 pairs, the second CTAs of their SMs stay away
    ([300, 290, 310, 280], 640, 200, torch.bfloat16),  # several sequences, pivots apart
    ([512] * 16, 768, 256, torch.bfloat16),            # every CTA works
    ([384] * 32, 512, 256, torch.bfloat16),            # 160 pairs: more than SMs
    ([320] * 30 + [40, 2], 384, 250, torch.float32),   # the same in fp32, small ones among them
    ([33, 95, 97, 65, 4000], 512, 60, torch.bfloat16), # half tiles that are partly filled, many tiles beside few
    ([5000], 256, 130, torch.float32),                 # 79 tiles: half tiles end where there are too many
    ([20000], 256, 130, torch.bfloat16),               # 313 tiles: whole ones
])
def test_extraction_of_batches(lengths, d, r, dtype):
    import paper_2403_02352_b200 as atp
    ranks = [min(r, L, d) for L in lengths]
    X = states(len(lengths) + d, lengths, d, 48, dtype)
    ctx = atp.Context(0)
    U, Xr, sigma = atp.atp_principal_basis(ctx, X, lengths, ranks)
    ctx.poll()
    f32 = dtype == torch.float32
    row = comp = 0
    for L, k in zip(lengths, ranks):
        x, u, xr = X[row:row + L].double(), U[row:row + L, :k].double(), Xr[comp:comp + k].double()
        s = sigma[comp:comp + k].double()
        row, comp = row + L, comp + k
        assert (u.T @ u - torch.eye(k, device="cuda")).abs().max() <= (5e-5 if f32 else 2e-2)
        assert (xr - u.T @ x).abs().max() <= 8 * (2.0 ** -23 if f32 else 2.0 ** -8) * s[0]
        n = torch.linalg.vector_norm(xr, dim=1)
        off = (xr @ xr.T / n[:, None] / n[None]).fill_diagonal_(0.0)
        assert off.abs().max() <= (1e-4 if f32 else 5e-2)
        assert bool((s[1:] <= s[:-1] + 1e-6 * s[0]).all())
    ctx.close()


@pytest.mark.parametrize("slow", [3e-5, 1e-4, 1e-3])
def test_pivots_of_graded_panels(slow):
    """Panels whose pivots fall over many orders, down to a few decades above the threshold of a dependent column: the chain of
    reciprocals in the factor has to keep the small ones (U^T U - I to fp32 rounding times the rotations of a row)."""
    import paper_2403_02352_b200 as atp
    gen = torch.Generator(device="cuda").manual_seed(7)
    L, d, r = 400, 512, 130
    u = torch.linalg.qr(torch.randn((L, L), generator=gen, device="cuda"))[0]
    v = torch.linalg.qr(torch.randn((d, L), generator=gen, device="cuda"))[0]
    X = (u * slow ** (torch.arange(L, device="cuda") / 64.0).clamp(max=1.0)) @ v.T
    ctx = atp.Context(0)
    U, _, _ = atp.atp_principal_basis(ctx, X, [L], [r])
    ctx.poll()
    U = U[:, :r].double()
    assert (U.T @ U - torch.eye(r, device="cuda")).abs().max() <= 5e-5
    ctx.close()
