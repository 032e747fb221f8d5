"""The codebook gradient of many scalar weights, whose sums have thousands of terms per thread (B200 only)."""
import pytest

pytestmark = pytest.mark.gpu


def reference(W, C, tau, G):
    """g_l = sum_i A_il G_i + (1 / tau) e_il(q) n_il in float64, q_ij = G_i c_j (the map of the codebook-gradient pass)."""
    import torch
    W, C = W[:, 0], C[:, 0].double()
    g, step = torch.zeros_like(C), max(1, (1 << 26) // C.numel())
    for a in range(0, W.numel(), step):
        w, Gc = W[a:a + step].double()[:, None], G[a:a + step].double()
        A = torch.softmax(-(w - C).abs() / tau, 1)
        q = Gc * C
        e = A * (q - (A * q).sum(1, keepdim=True)) / tau
        g += (A * Gc + e * torch.sign(w - C)).sum(0)
    return g


# weights of a thread: 221, 57, 900 and 3500
@pytest.mark.parametrize("m,k", [(1 << 26, 4), (1 << 24, 16), (20_000_003, 64), (1 << 24, 256)])
def test_sums_of_many_terms(m, k):
    """70 % of the weights share one value and dL/dWq has one sign, which is where a long fp32 sum would drift.  The
    exponential and the reciprocal are good to 2e-7 of a term each."""
    import torch
    from paper_2312_07759_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(k)
    W = torch.randn(m, 1, device="cuda", generator=g) * 0.03
    W = torch.where(torch.rand(m, 1, device="cuda", generator=g) < 0.7, torch.full_like(W, 0.011), W).contiguous()
    C0 = torch.linspace(-0.06, 0.06, k, device="cuda").reshape(k, 1)
    G = 0.3 + 0.05 * torch.randn(m, 1, device="cuda", generator=g)
    ctx = B.Context()
    C = ctx.forward(W, C0, 0.02, 0.0, 5).C
    dC = ctx.backward(G, B.JFB, 0.0, 0, 1.0, want_dW=False)[1][:, 0].double()
    ref = reference(W, C, 0.02, G)
    err = float((dC - ref).norm() / ref.norm())
    assert err < 4e-7
