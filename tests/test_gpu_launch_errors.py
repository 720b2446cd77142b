"""A launch that the runtime refuses is the call's error alone: nothing of it is left for the caller's next check."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_a_refused_launch_leaves_no_pending_error():
    from paper_2410_03090_b200 import binding as ub

    B, N, D = 66000, 2, 8                      # one grid row per sequence and head, 65535 at most
    ctx = ub.Context(ub.make_shape(B, 1, 1, 1, N, 128, 1, "bf16"))
    K = torch.zeros(B, 1, N, 128, dtype=torch.bfloat16, device="cuda")
    q = torch.zeros(B, 1, 128, dtype=torch.bfloat16, device="cuda")
    X = torch.zeros(B, N, D, dtype=torch.bfloat16, device="cuda")
    indices, Xout = torch.zeros(B, 1, dtype=torch.int32, device="cuda"), torch.zeros(B, 1, D, dtype=torch.bfloat16, device="cuda")
    one = torch.ones(4, device="cuda")
    torch.cuda.synchronize()
    with pytest.raises(RuntimeError):
        ub.uncomp_evict_hidden(ctx, q, K, X, 1, indices=indices, Xout=Xout)
    assert float((one + 1).sum()) == 8.0       # torch asks for the last error after each of its launches
    assert ub.uncomp_status(ctx) == 0
