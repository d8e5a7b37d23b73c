"""The tensor-core GEMM behind the low-rank linear layer and the attention projections, at the edges of its tiles: both
forms (one CTA, a pair of CTAs), partly filled tiles in M, N and K, one and many problems per launch, more tiles than CTAs.
Reference: the same formula in 64 bits on the GPU."""
import numpy as np
import pytest
import torch

from gpu_util import TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2403_02352_b200 as atp
    c = atp.Context(0)
    yield c
    c.close()


def _mat(g, rows, cols, scale):
    t = torch.zeros((rows, (cols + 7) // 8 * 8), dtype=torch.bfloat16, device="cuda")
    t[:, :cols] = (torch.randn((rows, cols), generator=g, device="cuda") * scale).bfloat16()
    return t[:, :cols]


@pytest.mark.parametrize("act", [None, "gelu", "swiglu"])
@pytest.mark.parametrize("lengths,ranks,d,d_out", [
    ([1], [1], 8, 1),                              # one element
    ([77], [19], 96, 127),                         # one tile, ragged
    ([128, 129, 5], [64, 65, 1], 65, 129),         # three problems, edges of 128
    ([1030], [257], 200, 4100),                    # pairs of CTAs, one row / column past a tile
    ([2047], [300], 72, 2049),                     # pairs, one short / one past
    ([1024, 511, 700], [130, 64, 63], 128, 3000),  # pairs, several problems
    ([300] * 17, [33] * 17, 64, 520),              # two launches (more problems than one carries)
    ([1300], [128], 64, 11008),                    # several tiles per CTA: both accumulators, stages wrap around
])
def test_linear_tile_edges(ctx, act, lengths, ranks, d, d_out):
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(sum(lengths) + d_out)
    rows, tr = sum(lengths), sum(ranks)
    U, X = _mat(g, rows, max(ranks), max(ranks) ** -0.5), _mat(g, tr, d, 1.0)
    W, Wg = _mat(g, d, d_out, d ** -0.5), _mat(g, d, d_out, d ** -0.5)
    bias = torch.randn(d_out, generator=g, device="cuda") if act != "swiglu" else None
    pad = torch.full((rows, (d_out + 7) // 8 * 8), 7.0, dtype=torch.bfloat16, device="cuda")
    Y = atp.atp_lowrank_linear(ctx, U, X, W, lengths, ranks, bias=bias, act=act, W_gate=Wg if act == "swiglu" else None,
                               out=pad[:, :d_out])
    ctx.poll()
    T, Tg = (X.double() @ W.double()).bfloat16().double(), (X.double() @ Wg.double()).bfloat16().double()
    ro = ko = 0
    for L, r in zip(lengths, ranks):
        u = U[ro:ro + L, :r].double()
        y = u @ T[ko:ko + r]
        if bias is not None:
            y = y + bias.double()
        if act == "gelu":
            y = torch.nn.functional.gelu(y)
        if act == "swiglu":
            y = torch.nn.functional.silu(u @ Tg[ko:ko + r]) * y
        err = float((Y[ro:ro + L].double() - y).abs().max() / y.abs().max().clamp_min(1e-6))
        assert err <= TOL["bf16"], (L, r, err)
        ro += L
        ko += r
    assert bool((pad[:, d_out:] == 7.0).all())     # the padding of the rows is not written


def test_extraction_products_in_both_forms(ctx):
    """The split products (two and three MMAs, transposed operands) at sizes that take pairs and single CTAs: the rows of
    X_r are U_r^T X up to the rounding of the stored basis."""
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(5)
    for L, d, r in ((700, 520, 40), (2100, 2056, 260)):
        k = 32
        X = (torch.randn((L, k), generator=g, device="cuda") * 0.8 ** torch.arange(k, device="cuda")) @ \
            torch.randn((k, d), generator=g, device="cuda") + 0.02 * torch.randn((L, d), generator=g, device="cuda")
        X = X.bfloat16()
        U, Xr, sig = atp.atp_principal_basis(ctx, X, [L], [r])
        ctx.poll()
        ref = U.double().T @ X.double()
        assert float((Xr.double() - ref).abs().max()) <= 8 * 2.0 ** -8 * float(sig[0])
        assert float((U.double().T @ U.double() - torch.eye(r, device="cuda", dtype=torch.double)).abs().max()) <= 2e-2
