"""Norm at the edges of its split of a row over threads: pieces of 16 bytes, 32 to 256 threads per row, partly filled
last pieces, the row-in-memory kernel behind them, residual and in-place output."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,cols", [("bf16", c) for c in (1, 7, 8, 9, 255, 1024, 1032, 2049, 4096, 8200, 16384, 16392)] +
                         [("f32", c) for c in (1, 3, 4, 5, 512, 516, 1027, 2048, 4097, 8192, 8196)])
@pytest.mark.parametrize("kind,residual,in_place", [("rms", False, False), ("layer", True, False), ("layer", True, True)])
def test_norm_edges(dtype, cols, kind, residual, in_place):
    import paper_2403_02352_b200 as atp
    ctx = atp.Context(0)
    rng = np.random.default_rng(cols)
    rows = 19                                              # not a multiple of the rows per CTA
    X = to_dev(rng.standard_normal((rows, cols)) * 3 + 1, dtype)
    R = to_dev(rng.standard_normal((rows, cols)), dtype) if residual else None
    ref = oracle.norm(to_np(X), residual=to_np(R) if residual else None, kind=kind)
    pad = X.as_strided((rows, X.stride(0)), (X.stride(0), 1))
    pad[:, cols:] = 7.0
    Y = X if in_place else torch.full_like(pad, 7.0)[:, :cols]
    out = atp.atp_input_norm(ctx, X, R, kind=kind, out=Y)
    # one rounding to the storage type (2^-9, 2^-24 relative to entries of at most ~5) and, in fp32, the row sums
    tol = 2.0 ** -8 if dtype == "bf16" else 2e-6
    assert np.abs(to_np(out) - ref).max() <= tol * max(np.abs(ref).max(), 1e-6)
    whole = Y.as_strided((rows, Y.stride(0)), (Y.stride(0), 1))
    assert bool((whole[:, cols:] == 7.0).all())            # the padding of the rows is not written
    ctx.close()


def test_norm_unaligned_fp32_rows():
    import paper_2403_02352_b200 as atp
    ctx = atp.Context(0)
    base = torch.randn((33, 101), device="cuda")
    X = base[:, 1:]                                        # 4-byte aligned rows: the row-in-memory kernel
    out = atp.atp_input_norm(ctx, X, None, kind="rms", out=torch.empty((33, 100), device="cuda"))
    assert np.abs(to_np(out) - oracle.norm(to_np(X), kind="rms")).max() <= 1e-5
    ctx.close()
