"""How the CTAs of the rotation and of the orthonormalisation are dealt out: batches on both sides of every line between the ways
(an SM for every CTA, pivots seated on SMs of their own with the CTAs beside them away, every CTA at work, more pairs of blocks than
SMs), the lengths derived from the number of SMs; iterates whose Gram matrix goes by half tiles, partly filled ones among them, and by
whole tiles."""
import pytest
import torch

from test_gpu_group_seats import states

pytestmark = pytest.mark.gpu


def way(pairs):
    """The way a batch goes, from the pairs of 32-row blocks of its sequences: the rule of the launch for two CTAs an SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    items = [p * (p + 1) // 2 + p * ((p + 1) // 2) for p in pairs]
    share = lambda workers, n: min(n, workers * n // sum(items))
    if sum(pairs) > sms:
        return "shared"
    if any(n > 2 * share(2 * sms - 2 * sum(pairs), n) for n in items):
        return "every CTA"
    used = sum(pairs) + sum(share(2 * sms - 2 * sum(pairs), n) for n in items)
    return "seated" if used > sms else "an SM each"


def check(X, lengths, ranks, f32):
    """Against 64 bits: U^T U to the storage type's rounding; singular values of the planted part to 1e-4 (bf16: 1e-3), as in the
    parity tests; rows of X_r as long as sigma says to the storage type's rounding, and orthogonal: what the rotation may leave
    (1e-6, 3e-4) plus five standard deviations of the rounding of two rows (2^-9 / sqrt(d) each at d >= 256); and U the leading
    subspace, within 5 % of the best residual and the rounding of U."""
    import paper_2403_02352_b200 as atp
    ctx = atp.Context(0)
    try:
        U, Xr, sigma = atp.atp_principal_basis(ctx, X, lengths, ranks)
        ctx.poll()
    finally:
        ctx.close()
    row = comp = 0
    for L, k in zip(lengths, ranks):
        x, u, xr = X[row:row + L].double(), U[row:row + L, :k].double(), Xr[comp:comp + k].double()
        s = sigma[comp:comp + k].double()
        row, comp = row + L, comp + k
        exact = torch.linalg.svdvals(x)
        lead = min(32, k, L // 2)
        assert (u.T @ u - torch.eye(k, device="cuda")).abs().max() <= (5e-5 if f32 else 2e-2)
        assert ((s - exact[:k]) / exact[:k])[:lead].abs().max() <= (1e-4 if f32 else 1e-3)
        n = torch.linalg.vector_norm(xr, dim=1)
        assert ((n - s) / s).abs().max() <= (1e-4 if f32 else 2.0 ** -8)
        off = (xr @ xr.T / n[:, None] / n[None]).fill_diagonal_(0.0)
        assert off.abs().max() <= (5e-6 if f32 else 1e-3)
        q = torch.linalg.qr(u)[0]
        left, best = (x - q @ (q.T @ x)).square().sum(), exact[k:].square().sum()
        assert left <= 1.05 ** 2 * best + ((2.0 ** -20 if f32 else 2.0 ** -9) ** 2) * x.square().sum()
        assert bool((s[1:] <= s[:-1] + 1e-6 * s[0]).all())


@pytest.mark.parametrize("lengths,d,r,dtype", [
    ([512], 512, 120, torch.float32),
    ([1500], 1600, 1000, torch.bfloat16),
    ([300, 290, 310, 280], 640, 200, torch.bfloat16),
    ([512] * 16, 768, 256, torch.bfloat16),
    ([384] * 32, 512, 256, torch.bfloat16),
    ([320] * 30 + [40, 2], 384, 250, torch.float32),
    ([33, 95, 97, 65, 4000], 512, 60, torch.bfloat16), # half tiles that are partly filled, many tiles beside few
    ([5000], 256, 130, torch.float32),
    ([20000], 256, 130, torch.bfloat16),               # 313 tiles: whole ones
])
def test_batches_against_64_bits(lengths, d, r, dtype):
    check(states(len(lengths) + d, lengths, d, 48, dtype), lengths, [min(r, L, d) for L in lengths], dtype == torch.float32)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("first,then", [("an SM each", "seated"), ("seated", "every CTA")])
def test_rotation_of_one_sequence_on_both_sides(first, then, dtype):
    p = next(p for p in range(1, 70) if way([p]) == first and way([p + 1]) == then)
    for pairs in (p, p + 1):
        L = 64 * pairs - 5
        check(states(pairs, [L], 64 * pairs + 48, 48, dtype), [L], [L - 70], dtype == torch.float32)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("more,expected", [(0, "every CTA"), (1, "shared")])
def test_rotation_of_as_many_pairs_as_sms(more, expected, dtype):
    total = torch.cuda.get_device_properties(0).multi_processor_count + more
    pairs = [total // 32 + (i < total % 32) for i in range(32)]
    assert sum(pairs) == total and way(pairs) == expected
    lengths = [64 * p - 3 for p in pairs]
    check(states(total, lengths, 400, 48, dtype), lengths, [L - 60 for L in lengths], dtype == torch.float32)


def test_rotation_of_one_large_sequence_among_small_ones():
    """Shares by size alone came to more CTAs than are resident here, and the call was refused."""
    lengths = [2112] + [64] * 31
    assert way([33] + [1] * 31) == "every CTA"
    check(states(1, lengths, 2176, 48, torch.bfloat16), lengths, [2048] + [40] * 31, False)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("beyond", [0, 1])
def test_gram_matrix_on_both_sides_of_half_tiles(beyond, dtype):
    """A sequence alone has two CTAs an SM: half tiles up to as many tiles as SMs, whole ones from the next row on."""
    L = 64 * torch.cuda.get_device_properties(0).multi_processor_count + beyond
    check(states(L, [L], 256, 48, dtype), [L], [100], dtype == torch.float32)
