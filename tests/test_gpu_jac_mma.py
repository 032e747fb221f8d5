"""The adjoint iteration on the Jacobian formed by the tensor cores (pairs and quadruples of weights, more than 8 centroids)
against the float64 oracle at the centroids the library returned, and its bounded waits (B200 only)."""
import numpy as np
import pytest

from parity_util import TOL_GRAD, assert_close

pytestmark = pytest.mark.gpu


def data(sizes, d, k, std, seed):
    rng = np.random.default_rng(seed)
    m = sum(sizes)
    W = (rng.standard_normal((m, d)) * std).astype(np.float32)
    offs = [0] + [int(x) for x in np.cumsum(sizes)]
    C0 = np.concatenate([W[a:b][rng.permutation(b - a)[:k]] for a, b in zip(offs, offs[1:])])
    G = (rng.standard_normal((m, d)) * 0.3 + 0.1).astype(np.float32)
    return W, C0, G, offs


# codebooks at the edges of the tiles (k d of 18, 64, 66 and 68, 128, 132, 256, 260, 512, 640, 1024; odd k), layers of fewer
# weights than one stage takes, of a stage and one weight, of several blocks, and batches of ragged layers
@pytest.mark.parametrize("d,k,sizes", [
    (2, 9, [9]), (2, 9, [129]), (2, 32, [20001]), (2, 33, [65]), (2, 33, [4097]), (2, 64, [50001]), (2, 65, [3001]), (2, 128, [20000]),
    (2, 129, [700]), (2, 256, [30011]), (4, 9, [40]), (4, 16, [128]), (4, 16, [90001]), (4, 17, [10000]), (4, 32, [30001]),
    (4, 33, [64]), (4, 33, [5003]), (4, 65, [6000]), (4, 128, [9001]), (4, 160, [2001]), (4, 256, [257]), (4, 256, [12001]),
    (4, 16, [1001, 37, 40003, 16, 9000]), (2, 24, [30001, 129, 24]), (4, 40, [3000, 65, 10001]), (2, 200, [4001, 200, 777]),
])
def test_adjoint_on_the_tensor_core_jacobian(d, k, sizes):
    import torch
    from oracle import idkm_ref as R
    from paper_2312_07759_b200 import binding as B
    iters, adj, alpha, tau = 60, 40, 0.25, float(np.float32(0.01))
    W, C0, G, offs = data(sizes, d, k, 0.03, d * 1000 + k)
    ctx = B.Context()
    Wd, Cd, Gd = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    fr = ctx.forward(Wd, Cd, tau, 0.0, iters, layer_offsets=offs)
    n0 = ctx.launches
    dW, dC = ctx.backward(Gd, B.IMPLICIT, 0.0, adj, alpha)
    torch.cuda.synchronize()
    assert ctx.launches - n0 == (3 if k * d <= 64 else 4)     # (the route is taken)
    info = ctx.info()
    assert ctx.busy_tickets() == 0
    for l, (a, b) in enumerate(zip(offs, offs[1:])):
        W64, G64 = W[a:b].astype(np.float64), G[a:b].astype(np.float64)
        C = fr.C.cpu().numpy()[l * k:(l + 1) * k].astype(np.float64)
        _, _, S, F = R.final(W64, C, tau)
        ri, ci, _, _ = R.backward(W64, G64, C, tau, S, F, mode="implicit", alpha=alpha, adj_max_iter=adj)
        assert info[l].status == 0 and info[l].adj_iters == adj
        assert_close(dC.cpu().numpy()[l * k:(l + 1) * k], ci, TOL_GRAD, f"layer {l} dC")
        assert_close(dW.cpu().numpy()[a:b], ri, TOL_GRAD, f"layer {l} dW")
    again = ctx.backward(Gd, B.IMPLICIT, 0.0, adj, alpha)
    assert torch.equal(again[0], dW) and torch.equal(again[1], dC)


@pytest.mark.parametrize("d,k", [(4, 12), (4, 48)])
def test_it_stops_at_the_tolerance_like_the_passes(d, k):
    import torch
    from paper_2312_07759_b200 import binding as B
    W, C0, G, _ = data([20000], d, k, 0.03, k)
    W, C0, G = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    out = []
    for method in (0, 1):
        ctx = B.Context()
        ctx.set_adjoint_method(method)
        ctx.forward(W, C0, 0.02, 1e-6, 200)
        dW, dC = ctx.backward(G, B.IMPLICIT, 1e-4, 100, 0.5)
        out.append((ctx.info()[0], dW.cpu().numpy(), dC.cpu().numpy()))
    assert out[0][0].status == out[1][0].status == 0
    assert out[0][0].adj_iters == out[1][0].adj_iters < 100
    assert_close(out[0][2], out[1][2], TOL_GRAD, "dC")
    assert_close(out[0][1], out[1][1], TOL_GRAD, "dW")


def test_a_lost_arrival_ends_the_iteration_with_a_status():
    """The blocks that iterate on the matrix wait a bounded time for one another; the next call is as before."""
    import torch
    from paper_2312_07759_b200 import binding as B
    W, C0, G, _ = data([5000], 4, 32, 0.03, 3)
    W, C0, G = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    ctx = B.Context()
    ctx.forward(W, C0, 0.01, 0.0, 5)
    good = ctx.backward(G, B.IMPLICIT, 0.0, 30, 0.25)[1].cpu().numpy()
    ctx.set_test_hooks(missing_arrivals=1, spin_limit_ticks=2000000)      # about a millisecond per wait
    try:
        ctx.backward(G, B.IMPLICIT, 0.0, 30, 0.25)
        torch.cuda.synchronize()
        assert ctx.info()[0].status == B.ERR_TIMEOUT
    finally:
        ctx.set_test_hooks(0, 0)
    ctx.forward(W, C0, 0.01, 0.0, 5)
    again = ctx.backward(G, B.IMPLICIT, 0.0, 30, 0.25)[1].cpu().numpy()
    assert ctx.info()[0].status == 0 and np.array_equal(again, good)


@pytest.mark.parametrize("d,k", [(2, 9), (4, 16)])
def test_a_stage_that_never_fills_ends_the_pass_with_a_status(d, k):
    """k d <= 64: the pass and the iteration are one launch.  A block whose wait for its operands ran out says so before it
    joins the others, and the block that iterates on their sums keeps the status."""
    import torch
    from paper_2312_07759_b200 import binding as B
    W, C0, G, _ = data([60000], d, k, 0.03, 5)
    W, C0, G = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    ctx = B.Context()
    ctx.forward(W, C0, 0.01, 0.0, 5)
    good = ctx.backward(G, B.IMPLICIT, 0.0, 30, 0.25)[1].cpu().numpy()
    ctx.set_test_hooks(missing_arrivals=1, spin_limit_ticks=2000000)      # about a millisecond per wait
    try:
        ctx.backward(G, B.IMPLICIT, 0.0, 30, 0.25)
        torch.cuda.synchronize()
        assert ctx.info()[0].status == B.ERR_TIMEOUT
    finally:
        ctx.set_test_hooks(0, 0)
    assert ctx.busy_tickets() == 0
    ctx.forward(W, C0, 0.01, 0.0, 5)
    again = ctx.backward(G, B.IMPLICIT, 0.0, 30, 0.25)[1].cpu().numpy()
    assert ctx.info()[0].status == 0 and np.array_equal(again, good)


@pytest.mark.parametrize("d,k,tau", [(4, 16, 0.002), (4, 64, 0.003), (2, 64, 0.002)])
def test_no_less_exact_than_the_passes(d, k, tau):
    """Sums of products on the tensor cores are cut, not rounded: what that takes from every entry of X^T Y does not cancel
    against the diagonal sums, and a cold softmax makes much of the difference.  Both routes against the float64 oracle, the
    mean over four layers; single layers scatter by a factor of about two."""
    import torch
    from oracle import idkm_ref as R
    from paper_2312_07759_b200 import binding as B
    err = {0: 0.0, 1: 0.0}
    for seed in range(4):
        W, C0, G, _ = data([40000], d, k, 0.03, seed)
        Wd, Cd, Gd = (torch.from_numpy(x).cuda() for x in (W, C0, G))
        for method in err:
            ctx = B.Context()
            ctx.set_adjoint_method(method)
            C = ctx.forward(Wd, Cd, tau, 0.0, 20).C.cpu().numpy().astype(np.float64)
            dC = ctx.backward(Gd, B.IMPLICIT, 0.0, 40, 0.25)[1].cpu().numpy()
            assert ctx.info()[0].status == 0
            W64 = W.astype(np.float64)
            _, _, S, F = R.final(W64, C, tau, want_Wq=False)
            _, u, _, _ = R.backward(W64, G.astype(np.float64), C, tau, S, F, alpha=0.25, adj_max_iter=40, want_dW=False)
            err[method] += float(np.linalg.norm(dC - u) / np.linalg.norm(u)) / 4
    assert err[0] <= 1.5 * err[1] + 1e-7, err


# as many blocks as the workspace rule lets iterate on matrices at a time (576, 384, 576), which have to be resident together
@pytest.mark.parametrize("d,k,layers", [(2, 256, 9), (4, 256, 3), (4, 192, 6)])
def test_the_largest_batches_keep_the_route(d, k, layers):
    import torch
    from paper_2312_07759_b200 import binding as B
    W, C0, G, offs = data([300 + 64 * l for l in range(layers)], d, k, 0.03, layers)
    W, C0, G = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    out = []
    for method in (0, 1):
        ctx = B.Context()
        ctx.set_adjoint_method(method)
        ctx.forward(W, C0, 0.02, 0.0, 8, layer_offsets=offs)
        n0 = ctx.launches
        dW, dC = ctx.backward(G, B.IMPLICIT, 0.0, 100, 0.25)
        out.append((ctx.launches - n0, dW.cpu().numpy(), dC.cpu().numpy(), [i.status for i in ctx.info()]))
    assert out[0][0] == 4 and out[1][0] == 102 and out[0][3] == out[1][3]
    if all(s == 0 for s in out[0][3]):
        assert_close(out[0][2], out[1][2], TOL_GRAD, "dC")
        assert_close(out[0][1], out[1][1], TOL_GRAD, "dW")


@pytest.mark.parametrize("d,k", [(4, 64), (2, 128)])
def test_a_layer_with_nothing_to_solve_ends_before_the_matrix(d, k):
    """tau above the weights' spread: every centroid is in the mean, and the first step of the iteration changes nothing."""
    import torch
    from paper_2312_07759_b200 import binding as B
    W, C0, G, offs = data([30000, 20000], d, k, 0.02, 1)
    W[30000:] *= 40.0                      # (the second layer does not collapse)
    C0[k:] *= 40.0
    W, C0, G = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    for layers in (1, 2):
        n = offs[layers]
        got = []
        for method in (0, 1):
            ctx = B.Context()
            ctx.set_adjoint_method(method)
            ctx.forward(W[:n], C0[:layers * k], 0.2, 0.0, 60, layer_offsets=offs[:layers + 1])
            dW, dC = ctx.backward(G[:n], B.IMPLICIT, 1e-5, 200, 0.5)
            got.append((dW.cpu().numpy(), dC.cpu().numpy(), [(i.status, i.adj_iters) for i in ctx.info()]))
        assert got[0][2][0][1] == got[1][2][0][1] <= 1
        if layers == 1:
            assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
        else:
            assert got[0][2][1][1] > 1 and abs(got[0][2][1][1] - got[1][2][1][1]) <= 1
            assert_close(got[0][1], got[1][1], TOL_GRAD, "dC")
