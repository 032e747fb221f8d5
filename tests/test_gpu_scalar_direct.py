"""Scalar weights whose bins would not pay -- a softmax far colder than the weights' range, outliers, many weights on few values --
are evaluated weight by weight by all blocks of their layer (B200 only)."""
import numpy as np
import pytest

from parity_util import TOL_C, assert_close
from test_gpu_scalar import check

pytestmark = pytest.mark.gpu


def weights(kind, m, rng):
    w = rng.standard_normal(m) * 0.03
    if kind == "cold":               # (tau of the case far below the range)
        return w
    if kind == "outlier":            # one weight far outside the rest
        w[m // 2] = 3000.0
    elif kind == "both":             # ... on both sides
        w[0], w[m - 1] = -800.0, 1e5
    elif kind == "two levels":
        lv = np.where(rng.random(m) < 0.5, 0.0125, -0.03125)
        w = np.where(rng.random(m) < 0.9, lv, w)
    elif kind == "one level":        # nearly all weights equal
        w = np.where(rng.random(m) < 0.99, 0.02, w)
    return w


# one block and many, a block's share of one and of many rounds; sums of a thread's own (k <= 100) for all and for some of the
# threads, and sums of a warp's; one barrier an iteration (k <= 32, few blocks) and two
@pytest.mark.parametrize("kind,m,k,tau", [
    ("cold", 40, 17, 5e-5), ("cold", 517, 31, 3e-5), ("cold", 16385, 4, 2e-5), ("cold", 16384, 17, 1e-5), ("outlier", 600, 1, 0.05),
    ("cold", 100003, 33, 2e-5), ("cold", 30001, 100, 1e-5), ("cold", 30001, 101, 1e-5), ("cold", 60001, 255, 1e-5), ("cold", 200003, 256, 2e-5),
    ("cold", 1 << 20, 5, 3e-5), ("cold", 1 << 21, 32, 5e-5),
    ("outlier", 4096, 4, 0.01), ("outlier", 70000, 5, 0.003), ("outlier", 300007, 64, 0.002), ("both", 33000, 3, 0.02), ("both", 50001, 8, 0.05),
    ("both", 20000, 32, 0.5), ("two levels", 9001, 2, 0.004), ("two levels", 400003, 24, 0.004), ("two levels", 150001, 128, 0.002),
    ("one level", 8192, 4, 0.01), ("one level", 250001, 7, 0.003),
])
def test_weight_by_weight_against_the_oracle(kind, m, k, tau):
    rng = np.random.default_rng(m + k)
    W = weights(kind, m, rng).astype(np.float32).reshape(m, 1)
    u = np.unique(W[np.abs(W) < 1.0])
    C0 = rng.choice(u, size=min(k, u.size), replace=False).reshape(-1, 1).astype(np.float32)
    check(W, C0, float(np.float32(tau)), 6, 5, alpha=0.5)


def test_both_kinds_of_layers_in_one_batch():
    rng = np.random.default_rng(3)
    kinds, sizes = ["cold", "outlier", "two levels", "cold", "both", "one level"], [4001, 70003, 90001, 9, 33, 40000]
    offs = [0] + [int(x) for x in np.cumsum(sizes)]
    W = np.concatenate([weights(a, n, rng) for a, n in zip(kinds, sizes)]).astype(np.float32).reshape(-1, 1)
    C0 = np.concatenate([rng.choice(np.unique(W[a:b][np.abs(W[a:b]) < 1.0]), 6, replace=False) for a, b in zip(offs, offs[1:])])
    ctx = check(W, C0.reshape(-1, 1).astype(np.float32), float(np.float32(0.01)), 7, 6, alpha=0.5, offs=offs)
    assert ctx.busy_tickets() == 0


def test_outliers_do_not_blur_the_rest():
    """Every weight by itself: an error of the bulk is invisible beside an outlier in a norm."""
    import torch
    from oracle import idkm_ref as R
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(1)
    W = weights("both", 40000, rng).astype(np.float32).reshape(-1, 1)
    C0 = W[1:9].copy()
    tau = float(np.float32(0.003))
    fr = B.Context().forward(torch.from_numpy(W).cuda(), torch.from_numpy(C0).cuda(), tau, 0.0, 8)
    Ct, _, _, _ = R.forward(W.astype(np.float64), C0.astype(np.float64), tau, 0.0, 8)
    C, Wq = fr.C.cpu().numpy(), fr.Wq.cpu().numpy()
    near = np.abs(Ct[:, 0]) < 1.0
    assert near.sum() >= 3
    assert_close(C[near], Ct[near], TOL_C, "C of the bulk")
    ref = R.final(W.astype(np.float64), C.astype(np.float64), tau)[0]
    bulk = np.abs(W[:, 0]) < 1.0
    assert_close(Wq[bulk], ref[bulk], TOL_C, "Wq of the bulk")


@pytest.mark.parametrize("kind,k", [("outlier", 4), ("outlier", 64), ("two levels", 16), ("two levels", 64)])
def test_the_time_does_not_depend_on_where_the_weights_lie(kind, k):
    """An iteration of 1 M weights: 3 to 170 ms where single lanes or warps walk through such bins, a few tens of microseconds
    by all blocks.  The bound leaves room for any clock."""
    import torch
    from paper_2312_07759_b200 import binding as B
    m, rng = 1 << 20, np.random.default_rng(k)
    W = torch.from_numpy(weights(kind, m, rng).astype(np.float32).reshape(m, 1)).cuda()
    C0 = torch.from_numpy((rng.standard_normal((k, 1)) * 0.03).astype(np.float32)).cuda()
    ctx = B.Context()
    ctx.forward(W, C0, 0.003, 0.0, 3)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    ctx.forward(W, C0, 0.003, 0.0, 13)
    b.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(b) < 5.0


@pytest.mark.parametrize("m,k", [(4096, 6), (100003, 6), (100003, 40)])
def test_it_stops_repeats_and_times_out_like_the_other_forms(m, k):
    import torch
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(m)
    W = torch.from_numpy(weights("outlier", m, rng).astype(np.float32).reshape(m, 1)).cuda()
    C0 = W[:k].clone()
    runs = []
    for method in (0, 0, 1):
        ctx = B.Context()
        ctx.set_forward_loop(method)
        fr = ctx.forward(W, C0, 0.004, 1e-5, 500)
        runs.append((fr.C.cpu().numpy(), fr.Wq.cpu().numpy(), ctx.info()[0].status, ctx.info()[0].fwd_iters, len(ctx.history(0))))
    assert np.array_equal(runs[0][0], runs[1][0]) and np.array_equal(runs[0][1], runs[1][1])
    assert runs[0][2:] == runs[1][2:] and runs[0][2] == runs[2][2] == 0 and runs[0][3] < 500 and abs(runs[0][3] - runs[2][3]) <= 1
    ctx = B.Context()
    ctx.set_test_hooks(missing_arrivals=1, spin_limit_ticks=2000000)
    ctx.forward(W, C0, 0.004, 0.0, 5)
    torch.cuda.synchronize()
    assert ctx.info()[0].status == B.ERR_TIMEOUT
    ctx.set_test_hooks(0, 0)
    fr = ctx.forward(W, C0, 0.004, 1e-5, 500)
    assert ctx.info()[0].status == 0 and np.array_equal(fr.C.cpu().numpy(), runs[0][0])
