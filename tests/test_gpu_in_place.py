"""The soft-quantised weights written over the weights themselves: the loop must have read them by then (B200 only)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,k,m", [(1, 4, 4096), (1, 7, 100003), (1, 24, 70001), (1, 256, 33000), (2, 4, 30001), (4, 16, 9000)])
def test_forward_into_its_own_weights(d, k, m):
    import torch
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(m)
    W = torch.from_numpy((rng.standard_normal((m, d)) * 0.03).astype(np.float32)).cuda()
    C0 = W[torch.from_numpy(rng.choice(m, k, replace=False)).cuda()].contiguous()
    tau, iters = float(np.float32(0.01)), 6
    ref = B.Context()
    fr = ref.forward(W, C0, tau, 0.0, iters)
    ctx = B.Context()
    nbytes = B.workspace_bytes(m, d, k, 1)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    X, C = W.clone(), torch.empty_like(C0)
    rc = ctx.forward_raw(X.data_ptr(), m, d, C0.data_ptr(), k, tau, 0.0, iters, C.data_ptr(), None, X.data_ptr(), ws.data_ptr(), nbytes)
    torch.cuda.synchronize()
    assert rc == B.OK
    ctx.n_layers = 1
    assert ctx.info()[0].status == 0 and ctx.info()[0].fwd_iters == iters
    # two ways of adding up the same fp32 terms: 1e-7 a step, six steps
    assert torch.allclose(C, fr.C, rtol=0, atol=2e-6 * float(fr.C.abs().max()))
    assert torch.allclose(X, fr.Wq, rtol=0, atol=2e-6 * float(fr.Wq.abs().max()))
