"""Extraction at the sizes where its tile and pairing logic can go wrong: projected sizes around the multiples of the
32-row blocks, the 64-column panels and the 64-row pivot blocks, single pair, odd pair counts, graded and flat spectra.
Every bound is the one of the parity tests (basis invariants against the oracle's spectrum)."""
import numpy as np
import pytest

import atp_inputs as ai
from gpu_util import basis_invariants, residual_ok, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2403_02352_b200 as atp
    c = atp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("sizes", [
    [(2, 1), (31, 9)],                 # one partly filled pair of blocks
    [(32, 20), (33, 33)],              # one block / one row more
    [(64, 40), (65, 1)],               # exactly one pivot block / the first row of the second
    [(96, 96), (97, 40), (127, 100)],  # odd number of blocks, partly filled last panel
    [(128, 128), (129, 70)],           # two pairs / three pairs with one row in the last
    [(300, 129), (193, 193)],          # three and four pairs
])
@pytest.mark.parametrize("decay", [0.6, 0.97])     # graded over many orders / nearly flat
def test_extraction_at_block_edges(ctx, dtype, sizes, decay):
    import paper_2403_02352_b200 as atp
    rng = np.random.default_rng(sum(L * r for L, r in sizes))
    d = 200
    xs = [ai.finish(ai.planted_matrix(rng, L, d, decay ** np.arange(min(L, 48)), 0.02)[0], dtype) for L, _ in sizes]
    lengths, ranks = [L for L, _ in sizes], [r for _, r in sizes]
    U, Xr, sig = atp.atp_principal_basis(ctx, to_dev(np.concatenate(xs), dtype), lengths, ranks)
    ctx.poll()
    U, Xr, sig = to_np(U), to_np(Xr), to_np(sig.reshape(-1, 1)).ravel()
    ro, ko = np.concatenate([[0], np.cumsum(lengths)]), np.concatenate([[0], np.cumsum(ranks)])
    for b, X in enumerate(xs):
        inv = basis_invariants(X, U[ro[b]:ro[b + 1], :ranks[b]], Xr[ko[b]:ko[b + 1]], sig[ko[b]:ko[b + 1]])
        assert inv["orth"] <= (5e-5 if dtype == "f32" else 2e-2), (b, inv["orth"])
        assert inv["offdiag"] <= (1e-4 if dtype == "f32" else 5e-2), (b, inv["offdiag"])
        assert inv["xr_vs_utx"] <= 8 * (2.0 ** -23 if dtype == "f32" else 2.0 ** -8), (b, inv["xr_vs_utx"])
        assert residual_ok(inv["res_sub"], inv["opt"], inv["normX"], dtype, 3e-2), (b, inv["res_sub"], inv["opt"])
        assert inv["sorted"]
