"""The stream a call of the binding runs on when none is given: the current device's current one."""
import pytest

import absorber_inputs as ai

pytestmark = pytest.mark.gpu


def test_calls_without_a_stream_use_the_current_one():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_15420_gb300 import build
    build.build()
    from paper_2607_15420_gb300 import binding as B
    assert B._stream(None) == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert B._stream(None) == side.cuda_stream
        with torch.cuda.stream(torch.cuda.default_stream()):
            assert B._stream(None) == torch.cuda.default_stream().cuda_stream
        assert B._stream(None) == side.cuda_stream
        # a fill queued on the stream before the call is what the call reads
        prob = B.Problem(ai.PARAMS, ai.make_feeds(2000, 1))
        x = torch.empty(prob.n_primal, dtype=torch.float64, device="cuda")
        big = torch.ones(1 << 27, device="cuda")
        for _ in range(4):
            big.mul_(1.0)
        x.fill_(0.9)
        c = torch.zeros(prob.n_row, dtype=torch.float64, device="cuda")
        prob.eval_grad_jac_hess(x, c=c)
    side.synchronize()
    ref = torch.zeros_like(c)
    prob.eval_grad_jac_hess(x, c=ref)
    torch.cuda.synchronize()
    assert torch.equal(c.view(-1, prob.ld)[:, :2000], ref.view(-1, prob.ld)[:, :2000])
    assert B._stream(None) == torch.cuda.current_stream().cuda_stream
