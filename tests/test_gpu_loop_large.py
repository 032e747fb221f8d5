"""The one-launch forward loop of the larger codebooks (pairs of weights: more than 16 centroids, quadruples: more than 8) against
the float64 oracle, both distances and collapsing layers, and its bounded waits (B200 only)."""
import numpy as np
import pytest

from parity_util import TOL_C, assert_close

pytestmark = pytest.mark.gpu


def draw(sizes, d, k, std, seed):
    rng = np.random.default_rng(seed)
    W = (rng.standard_normal((sum(sizes), d)) * std).astype(np.float32)
    offs = [0] + [int(x) for x in np.cumsum(sizes)]
    C0 = np.concatenate([W[a:b][rng.permutation(b - a)[:k]] for a, b in zip(offs, offs[1:])])
    return W, C0, offs


def check(sizes, d, k, tau, iters, std=0.03, squared=False, tol=0.0):
    import torch
    from oracle import idkm_ref as R
    from paper_2312_07759_b200 import binding as B
    W, C0, offs = draw(sizes, d, k, std, 7 * d + k)
    ctx = B.Context()
    ctx.set_distance(squared)
    Wd, Cd = torch.from_numpy(W).cuda(), torch.from_numpy(C0).cuda()
    n0 = ctx.launches
    fr = ctx.forward(Wd, Cd, tau, tol, iters, layer_offsets=offs)
    torch.cuda.synchronize()
    assert ctx.launches - n0 == 3     # (the route is taken: start, loop, final pass)
    info = ctx.info()
    C = fr.C.cpu().numpy()
    for l, (a, b) in enumerate(zip(offs, offs[1:])):
        with R.squared_distance(squared):
            Ct, n, _, _ = R.forward(W[a:b].astype(np.float64), C0[l * k:(l + 1) * k].astype(np.float64), tau, tol, iters)
        assert info[l].fwd_iters == n
        assert_close(C[l * k:(l + 1) * k], Ct, TOL_C, f"layer {l} C")
    again = ctx.forward(Wd, Cd, tau, tol, iters, layer_offsets=offs)
    assert torch.equal(again.C, fr.C)


# codebooks at the edges of the kernels' sizes and odd ones; fewer weights than a block takes, one more than a set, sizes at
# which every block adds all partials and at which it adds a share
SHAPES = [
    (2, 17, [17]), (2, 17, [4099]), (2, 32, [129]), (2, 32, [70001]), (2, 33, [9001]), (2, 64, [64]), (2, 64, [130003]), (2, 65, [5000]),
    (2, 128, [20001]), (4, 9, [9]), (4, 9, [1000]), (4, 16, [150001]), (4, 17, [4097]), (4, 32, [60000]), (4, 33, [33]),
    (4, 33, [1025]), (4, 64, [50007]), (4, 65, [129]), (4, 128, [12001]), (4, 129, [3001]), (4, 256, [256]), (4, 256, [20003]),
]


@pytest.mark.parametrize("d,k,sizes", SHAPES + [
    (2, 129, [9000]), (2, 256, [40001])])
def test_loop_against_the_oracle(d, k, sizes):
    check(sizes, d, k, float(np.float32(0.01)), 5)


@pytest.mark.parametrize("d,k,sizes", SHAPES)
def test_squared_distance(d, k, sizes):
    check(sizes, d, k, float(np.float32(4e-4)), 4, squared=True)


@pytest.mark.parametrize("d,k,sizes", [(2, 20, [5001]), (2, 64, [20001]), (2, 256, [3000]), (4, 12, [7001]), (4, 32, [30000]), (4, 64, [4001]),
                                       (4, 256, [9001])])
def test_collapsing_layers(d, k, sizes):
    """tau far above the weights' spread: the centroids fall together and the increment form takes over."""
    check(sizes, d, k, 0.5, 8)


def test_it_ends_at_a_tolerance():
    check([20001], 4, 20, float(np.float32(0.02)), 60, tol=2e-3)


@pytest.mark.parametrize("d,k", [(2, 40), (4, 12), (4, 100)])
def test_a_lost_arrival_ends_the_loop_with_a_status(d, k):
    import torch
    from paper_2312_07759_b200 import binding as B
    W, C0, _ = draw([6000], d, k, 0.03, k)
    W, C0 = torch.from_numpy(W).cuda(), torch.from_numpy(C0).cuda()
    ctx = B.Context()
    good = ctx.forward(W, C0, 0.01, 0.0, 5).C.cpu().numpy()
    ctx.set_test_hooks(missing_arrivals=1, spin_limit_ticks=2000000)      # about a millisecond per wait
    try:
        ctx.forward(W, C0, 0.01, 0.0, 5)
        torch.cuda.synchronize()
        assert ctx.info()[0].status == B.ERR_TIMEOUT and ctx.info()[0].fwd_iters == 0
    finally:
        ctx.set_test_hooks(0, 0)
    assert np.array_equal(ctx.forward(W, C0, 0.01, 0.0, 5).C.cpu().numpy(), good)
