"""What idkm_last_route says against the launches that a call makes (B200 only)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,d,k,layers,loop,adjoint,forward,backward", [
    (20000, 1, 4, 1, 0, 0, "interval form", "interval sums"),
    (20000, 1, 40, 3, 0, 1, "interval form", "fused passes"),
    (20000, 1, 16, 1, 1, 2, "a launch per iteration", "exact solve on the explicit Jacobian"),
    (20000, 2, 4, 2, 0, 0, "one-launch loop", "explicit Jacobian in registers"),
    (20000, 4, 8, 1, 0, 0, "one-launch loop", "explicit Jacobian in tiles"),
    (20000, 4, 16, 1, 0, 0, "one-launch loop of larger codebooks", "explicit Jacobian from the tensor cores"),
    (20000, 4, 16, 4, 0, 0, "a launch per iteration", "explicit Jacobian from the tensor cores"),
    (6000, 4, 256, 4, 0, 0, "a launch per iteration", "fused passes"),
])
def test_the_route_that_was_taken(m, d, k, layers, loop, adjoint, forward, backward):
    import torch
    from paper_2312_07759_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(k)
    W = torch.randn(m * layers, d, device="cuda", generator=g) * 0.03
    offs = [m * l for l in range(layers + 1)]
    C0 = torch.cat([W[a:a + k] for a in offs[:-1]]).contiguous()
    ctx = B.Context()
    ctx.set_forward_loop(loop)
    ctx.set_adjoint_method(adjoint)
    n0 = ctx.launches
    ctx.forward(W, C0, 0.02, 0.0, 20, layer_offsets=offs)
    n1 = ctx.launches
    assert ctx.last_route() == {"forward": forward, "adjoint": "none"}
    ctx.backward(torch.ones_like(W), B.IMPLICIT, 0.0, 40, 0.25)
    n2 = ctx.launches
    assert ctx.last_route() == {"forward": forward, "adjoint": backward}
    assert (n1 - n0 >= 20) == (forward == "a launch per iteration")
    assert (n2 - n1 >= 40) == (backward == "fused passes")
    ctx.backward(torch.ones_like(W), B.JFB, 0.0, 0, 1.0)
    assert ctx.last_route()["adjoint"] == "none"


@pytest.mark.parametrize("m,d,k,forward", [
    (13_000_000, 2, 128, "one-launch loop of larger codebooks"), (14_000_000, 2, 128, "a launch per iteration"),
    (3_000_000, 4, 32, "one-launch loop of larger codebooks"), (3_100_000, 4, 32, "a launch per iteration"),
])
def test_large_layers(m, d, k, forward):
    import torch
    from paper_2312_07759_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(k)
    W = torch.randn(m, d, device="cuda", generator=g) * 0.03
    ctx = B.Context()
    C = ctx.forward(W, W[:k].contiguous(), 0.01, 0.0, 3, want_Wq=False).C
    assert ctx.last_route()["forward"] == forward
    ctx.set_forward_loop(1)
    ref = ctx.forward(W, W[:k].contiguous(), 0.01, 0.0, 3, want_Wq=False).C
    assert float((C - ref).norm() / ref.norm()) < 1e-5


@pytest.mark.parametrize("k,iters,forward", [(4, 4, "one-launch loop"), (4, 5, "interval form"), (8, 4, "one-launch loop"), (9, 4, "interval form")])
def test_few_iterations_do_without_bins(k, iters, forward):
    import torch
    from paper_2312_07759_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(k)
    W = torch.randn(30000, 1, device="cuda", generator=g) * 0.03
    ctx = B.Context()
    C = ctx.forward(W, W[:k].contiguous(), 0.01, 0.0, iters).C
    assert ctx.last_route()["forward"] == forward
    ctx.set_forward_loop(1)
    ref = ctx.forward(W, W[:k].contiguous(), 0.01, 0.0, iters).C
    assert float((C - ref).norm() / ref.norm()) < 1e-5


# either side of the lines between the loop over few cold weights and the interval form: rows, centroids, iterations, tau
@pytest.mark.parametrize("m,k,iters,tau,forward", [
    (2048, 4, 30, 0.029, "one-launch loop"), (2048, 4, 30, 0.031, "interval form"), (2049, 4, 30, 0.0024, "one-launch loop"),
    (2049, 4, 5, 0.0026, "interval form"), (4096, 4, 30, 0.0024, "one-launch loop"), (4096, 2, 30, 0.0026, "interval form"),
    (2048, 5, 30, 9.9e-4, "one-launch loop"), (2048, 16, 30, 1.1e-3, "interval form"), (2049, 5, 30, 6.9e-4, "one-launch loop"),
    (4096, 16, 20, 7.1e-4, "interval form"), (4096, 16, 19, 7.1e-4, "one-launch loop"), (4097, 4, 20, 5e-4, "interval form"),
    (4097, 12, 20, 4.9e-4, "one-launch loop"), (16384, 12, 19, 9.9e-4, "one-launch loop"), (16384, 13, 20, 6.9e-4, "one-launch loop"),
    (16384, 16, 20, 7.1e-4, "interval form"), (16385, 3, 20, 1e-4, "interval form"), (16384, 17, 20, 1e-4, "interval form"),
])
def test_few_cold_weights(m, k, iters, tau, forward):
    import torch
    from paper_2312_07759_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(m + k)
    W = torch.randn(m, 1, device="cuda", generator=g) * 0.03
    C0 = torch.sort(W[:, 0])[0][((torch.arange(k, device="cuda") + 0.5) * m / k).long()].reshape(k, 1).contiguous()
    ctx = B.Context()
    C = ctx.forward(W, C0, tau, 0.0, iters).C
    assert ctx.last_route()["forward"] == forward
    ctx.set_forward_loop(1)
    ref = ctx.forward(W, C0, tau, 0.0, iters).C
    assert float((C - ref).norm() / ref.norm()) < 1e-5
