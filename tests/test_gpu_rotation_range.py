"""Extraction of inputs at other scales. A power of two changes no rounding of X, of the iterates or of the Gram matrix,
so the basis of 2^k X is that of X and its singular values are 2^k times those of X; what may differ are the scale factors
inside the kernels. The scales put the entries of the Gram matrix near 1e-18, where squares of its entries fall below
fp32's normal range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,k", [("f32", -20), ("f32", -26), ("f32", -28), ("f32", 20),
                                     ("bf16", -20), ("bf16", -26), ("bf16", -28), ("bf16", -30), ("bf16", 20)])
def test_scaled_input(dtype, k):
    import atp_inputs as ai
    import paper_2403_02352_b200 as atp
    from gpu_util import to_dev
    L, d, r = 384, 256, 96
    X = ai.finish(ai.planted_matrix(np.random.default_rng(3), L, d, 0.93 ** np.arange(64), 0.01)[0], dtype)
    c = atp.Context(0)
    try:
        x = to_dev(X, dtype)
        U, Xr, sig = atp.atp_principal_basis(c, x * 2.0 ** k, [L], [r])
        c.poll()
        u, xr = U.double(), Xr.double() * 2.0 ** -k
        exact = torch.linalg.svdvals(x.double())[:r]
        # the bounds of the parity tests: orthonormality, X_r = U^T X to the storage type, and the planted singular values
        # (those of the noise behind them are the range finder's)
        eps = 2.0 ** -23 if dtype == "f32" else 2.0 ** -8
        assert (u.T @ u - torch.eye(r, device="cuda")).abs().max().item() <= (5e-5 if dtype == "f32" else 2e-2)
        assert (xr - u.T @ x.double()).abs().max().item() <= 8 * eps * exact[0].item()
        assert ((sig.double() * 2.0 ** -k - exact) / exact)[:32].abs().max().item() <= (1e-4 if dtype == "f32" else 1e-3)
    finally:
        c.close()
