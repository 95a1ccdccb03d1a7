"""The library beside other work: a second stream of the caller while a long kernel runs and the next one waits for it."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_a_waiting_kernel_leaves_room_for_another_stream():
    """A forward pass of several milliseconds with the column sums queued behind it: a small kernel of another stream, which fits
    beside the forward's CTAs, runs while the forward does (the CTAs of the column sums come up near its end and do not
    take that room for all its length)."""
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    B, D, H = 65536, 8192, 8192
    A = torch.zeros(B, D, dtype=bf, device="cuda")
    W = torch.zeros(D, H, dtype=bf, device="cuda")
    out, db = torch.empty(B, H, dtype=bf, device="cuda"), torch.empty(H, device="cuda")
    ws = torch.empty(rad.rad_input_grad_workspace(B, H), dtype=torch.uint8, device="cuda")
    y = torch.ones(1 << 20, device="cuda")
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    begin, done, beside = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    for _ in range(2):                       # the first turn loads the kernels
        torch.cuda.synchronize()
        with torch.cuda.stream(main):
            begin.record()
            rad.rad_linear_forward(A, W, None, "none", out_act=out)
            rad.rad_linear_input_grad(out, W, db=db, workspace=ws)
            done.record()
        time.sleep(1e-3)
        with torch.cuda.stream(side):
            y.add_(1)
            beside.record()
        torch.cuda.synchronize()
    assert begin.elapsed_time(done) > 3.0
    assert begin.elapsed_time(beside) < 0.7 * begin.elapsed_time(done)
