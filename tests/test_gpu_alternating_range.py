"""Algorithm 1 over the range of its input: scales up to where the squares of u leave fp32 and down to where they leave
even a shifted fp64 product, and entries that are no numbers. The reference is the method with every dot product in
64 bits and R, u, v rounded to 32 bits where the library holds them; the library adds in another order, so u and v may
round the other way (2^-24 per round and element, a few of them per component)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def algorithm1(X, V0, r, inner):
    R, us, xs = X.float().clone(), [], []
    zero = torch.zeros((), device="cuda", dtype=torch.float64)
    for i in range(r):
        v = V0[i].float()
        for _ in range(inner):
            vv = v.double().square().sum()
            u = torch.where(vv > 0, (R.double() @ v.double()) / vv, zero).float()
            uu = u.double().square().sum()
            v = torch.where(uu > 0, (R.double().T @ u.double()) / uu, zero).float()
        n = uu.sqrt()
        us.append(torch.where(n > 0, u.double() / n, zero).float())
        xs.append((v.double() * n).float())
        R = R - u[:, None] * v[None, :]
    return torch.stack(us, 1), torch.stack(xs)


@pytest.mark.parametrize("L,d", [(64, 64), (50, 77), (700, 130)])
@pytest.mark.parametrize("k", [-100, -90, -83, -75, -60, 0, 60, 100])
def test_scales(L, d, k):
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(L + d)
    X = torch.randn((L, d), generator=g, device="cuda") * 2.0 ** k
    V0 = torch.randn((4, d), generator=g, device="cuda")
    c = atp.Context(0)
    try:
        U, W = atp.atp_alternating_basis(c, X, V0, [L], [4])
        c.poll()
        u, w = algorithm1(X, V0, 4, 2)
        assert (U - u).norm() <= 4e-6 * u.norm()
        assert (W.double() - w.double()).norm() <= 4e-6 * w.double().norm()
    finally:
        c.close()


@pytest.mark.parametrize("inner", [1, 2])
@pytest.mark.parametrize("col", [4, 5, 6, 7])
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan")])
def test_no_numbers(value, col, inner):
    # whatever the column, the component is what 64-bit arithmetic gives: u infinite or NaN, and nothing finite from then on
    # but the zeros that a vanishing or undefined |u|^2 stands for
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((64, 64), generator=g, device="cuda")
    X[3, col] = value
    V0 = torch.randn((3, 64), generator=g, device="cuda")
    c = atp.Context(0)
    try:
        U, W = atp.atp_alternating_basis(c, X, V0, [64], [3], inner=inner)
        c.poll()
        u, w = algorithm1(X, V0, 3, inner)
        for got, want in ((U, u), (W, w)):
            assert (got.isfinite() == want.isfinite()).all()
            assert torch.allclose(got.nan_to_num(0.0, 0.0, 0.0), want.nan_to_num(0.0, 0.0, 0.0), rtol=1e-5, atol=1e-6)
    finally:
        c.close()


def test_overflow_of_the_deflation():
    # finite input whose deflation leaves fp32: R becomes infinite in the course of the call
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randn((40, 36), generator=g, device="cuda").sign() * 3e38
    V0 = torch.randn((3, 36), generator=g, device="cuda")
    c = atp.Context(0)
    try:
        U, W = atp.atp_alternating_basis(c, X, V0, [40], [3])
        c.poll()
        u, w = algorithm1(X, V0, 3, 2)
        assert (U.isfinite() == u.isfinite()).all() and (W.isfinite() == w.isfinite()).all()
    finally:
        c.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("lengths,d", [
    ([48, 70], 28376), ([48, 70], 28408),      # the vectors of a CTA just fit in shared memory / no longer do
    ([5, 33], 40008), ([64], 60000),           # long rows
    ([80000] * 32, 16),                        # many rows to a CTA: u alone is near the shared memory
    ([130000] * 32, 8),                        # and beyond it
])
def test_vectors_beyond_shared_memory(lengths, d, dtype):
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(d)
    ranks = [2] * len(lengths)
    X = torch.randn((sum(lengths), d), generator=g, device="cuda").to(dtype)
    V0 = torch.randn((sum(ranks), d), generator=g, device="cuda")
    c = atp.Context(0)
    try:
        U, W = atp.atp_alternating_basis(c, X, V0, lengths, ranks)
        c.poll()
        eps = 4e-6 if dtype == torch.float32 else 2.0 ** -8          # bf16: the outputs' own rounding
        row = 0
        for b, L in enumerate(lengths):
            if b in (0, len(lengths) - 1):
                u, w = algorithm1(X[row:row + L], V0[2 * b:2 * b + 2], 2, 2)
                assert (U[row:row + L].float() - u).norm() <= eps * u.norm()
                assert (W[2 * b:2 * b + 2].float() - w).norm() <= eps * w.norm()
            row += L
    finally:
        c.close()
