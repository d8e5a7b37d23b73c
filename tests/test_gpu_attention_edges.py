"""The fused attention kernel at the edges of its tiles: one and two query tiles per CTA, rows past the last tile, partly
filled key blocks, and logits small enough for the single product of the scores or large enough for all three.
Reference: the same formula in 64 bits on the GPU."""
import math

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


@pytest.mark.parametrize("spread,decay", [(0.05, 1.0), (12.0, 1.0), (3.0, 0.99)])    # of the logits; of the keys, by row
@pytest.mark.parametrize("heads,dh", [(2, 128), (3, 64)])
@pytest.mark.parametrize("lengths,ranks", [
    ([1], [1]),
    ([128, 129, 256, 257], [127, 128, 129, 257]),
    ([385, 31, 640], [384, 31, 513]),                            # a single tile last; more blocks than the ring holds
])
def test_attention_tile_edges(ctx, lengths, ranks, heads, dh, spread, decay):
    import paper_2403_02352_b200 as atp
    g = torch.Generator(device="cuda").manual_seed(sum(lengths) + dh)
    randn = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float64)
    d, dp, rows = 520, heads * dh, sum(lengths)
    U = torch.zeros((rows, (max(ranks) + 7) // 8 * 8), dtype=torch.bfloat16, device="cuda")[:, :max(ranks)]
    X = torch.empty((sum(ranks), d), dtype=torch.bfloat16, device="cuda")
    ro = ko = 0
    for L, r in zip(lengths, ranks):
        U[ro:ro + L, :r] = torch.linalg.qr(randn(L, r))[0].bfloat16()
        X[ko:ko + r] = (randn(r, d) * math.sqrt(L / r) * decay ** torch.arange(r, device="cuda")[:, None]).bfloat16()
        ro, ko = ro + L, ko + r
    WQ, WK, WV = [(randn(d, dp) * (f / math.sqrt(d))).bfloat16() for f in (spread, 1.0, 1.0)]
    O = atp.atp_attention(ctx, None, U, X, WQ, WK, WV, heads, lengths, ranks)
    ctx.poll()
    ro = ko = 0
    for L, r in zip(lengths, ranks):
        u, x = U[ro:ro + L, :r].double(), X[ko:ko + r].double()
        split = lambda t: t.reshape(-1, heads, dh).transpose(0, 1)
        q, k, v = split(u @ (x @ WQ.double())), split(x @ WK.double()), split(x @ WV.double())
        ref = (torch.softmax(q @ k.transpose(1, 2) / math.sqrt(dh), -1) @ v).transpose(0, 1).reshape(L, dp)
        err = float((O[ro:ro + L].double() - ref).abs().max() / ref.abs().max())
        assert err <= TOL["bf16"], (L, r, err)
        ro, ko = ro + L, ko + r
