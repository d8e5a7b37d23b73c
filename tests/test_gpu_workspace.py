"""Every call runs in exactly the workspace its query names, writes nothing behind it, and refuses less."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
GUARD = 1 << 16


def inputs(dtype, lengths, ranks, d, d_out):
    import atp_inputs as ai
    from gpu_util import to_dev
    rng = np.random.default_rng(0)
    t = lambda r, c: to_dev(ai.finish(rng.standard_normal((r, c)) / c ** 0.5, dtype), dtype)
    q = [np.linalg.qr(rng.standard_normal((L, r)))[0] for L, r in zip(lengths, ranks)]
    U = np.concatenate([np.pad(u, ((0, 0), (0, max(ranks) - u.shape[1]))) for u in q])
    return t(sum(lengths), d), to_dev(ai.finish(U, dtype), dtype), t(sum(ranks), d), [t(d, d_out) for _ in range(3)]


def w48(W):
    """Columns of as many heads of 48 as there is room for."""
    return W[0].shape[1] // 48 * 48


CALLS = {
    "basis": lambda atp, c, X, U, Xr, W, n, r: atp.atp_principal_basis(c, X, n, r, auto_workspace=False),
    "basis_one_sided": lambda atp, c, X, U, Xr, W, n, r: atp.atp_principal_basis(c, X, n, r, auto_workspace=False, jacobi_block=1),
    "attention": lambda atp, c, X, U, Xr, W, n, r: atp.atp_attention(c, X, U, Xr, *W, W[0].shape[1] // 64, n, r, auto_workspace=False),
    "attention_rope": lambda atp, c, X, U, Xr, W, n, r: atp.atp_attention(c, X, U, Xr, *W, W[0].shape[1] // 64, n, r, rope_base=1e4,
                                                                         q_mode="full", auto_workspace=False),
    "attention_rope_48": lambda atp, c, X, U, Xr, W, n, r: atp.atp_attention(c, X, U, Xr, *[w[:, :w48(W)].contiguous() for w in W],
                                                                            w48(W) // 48, n, r, rope_base=1e4, auto_workspace=False),
    "swiglu": lambda atp, c, X, U, Xr, W, n, r: atp.atp_lowrank_linear(c, U, Xr, W[0], n, r, act="swiglu", W_gate=W[1], auto_workspace=False),
    "alternating": lambda atp, c, X, U, Xr, W, n, r: atp.atp_alternating_basis(c, X, torch.ones((sum(r), X.shape[1]), device="cuda").tril(),
                                                                              n, r, auto_workspace=False),
}


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("call", list(CALLS))
@pytest.mark.parametrize("lengths,ranks,d,d_out", [([96], [20], 72, 64), ([200, 130], [50, 64], 192, 320), ([700], [90], 512, 384)])
def test_exact_workspace(call, dtype, lengths, ranks, d, d_out):
    import paper_2403_02352_b200 as atp
    from paper_2403_02352_b200 import binding as B
    args = (*inputs(dtype, lengths, ranks, d, d_out), lengths, ranks)
    op = {"b": B.OP_BASIS, "a": B.OP_ATTENTION, "s": B.OP_LINEAR}[call[0]] if call != "alternating" else B.OP_ALTERNATING
    c = atp.Context(0)
    try:
        width = d_out // 48 * 48 if call == "attention_rope_48" else d_out
        n = (c.workspace_bytes(op, B.SeqDesc(lengths, ranks), d, width, B.F32 if dtype == "f32" else B.BF16) + 255) // 256 * 256
        c.set_workspace(torch.zeros(4 * n + GUARD, dtype=torch.uint8, device="cuda"))
        want = CALLS[call](atp, c, *args)
        buf = torch.full((n + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
        c.set_workspace(buf[:n])
        got = CALLS[call](atp, c, *args)
        c.poll()
        assert (buf[n:] == 0xA5).all()
        for a, b in zip(want if isinstance(want, tuple) else (want,), got if isinstance(got, tuple) else (got,)):
            assert torch.equal(a, b)
        c.set_workspace(buf[:256])
        with pytest.raises(atp.AtpError):
            CALLS[call](atp, c, *args)
    finally:
        c.close()
