"""Scalar weights in the interval form (bins with moments in the loop, one search per weight in the passes, the adjoint
iteration on interval sums) against the float64 oracle (B200 only).  The backward is compared at the centroids the library
itself returned, where no weight can lie between the two sides' centroids."""
import numpy as np
import pytest

from paper_2312_07759_b200 import workloads as WL
from parity_util import TOL_C, TOL_GRAD, assert_close

pytestmark = pytest.mark.gpu


def weights(kind, m, rng):
    if kind == "normal":
        return rng.standard_normal(m) * 0.03
    if kind == "laplace":
        return rng.laplace(0.0, 0.02, m)
    if kind == "pruned":            # half the weights are exactly zero
        return np.where(rng.random(m) < 0.5, 0.0, rng.standard_normal(m) * 0.03)
    if kind == "levels":            # three quarters of the weights sit on two values: bins of very many equal weights
        return np.where(rng.random(m) < 0.75, np.where(rng.random(m) < 0.5, 0.0125, -0.03125), rng.standard_normal(m) * 0.03)
    if kind == "offset":            # a narrow range far from zero
        return 1.0 + rng.standard_normal(m) * 1e-3
    if kind == "outlier":           # one weight far outside the rest
        w = rng.standard_normal(m) * 0.03
        w[m // 2] = 4.0
        return w
    raise ValueError(kind)


def check(W, C0, tau, iters, adj_iters, alpha=1.0, offs=None):
    import torch
    from oracle import idkm_ref as R
    from paper_2312_07759_b200 import binding as B
    m = W.shape[0]
    offs = [0, m] if offs is None else offs
    L = len(offs) - 1
    k = C0.shape[0] // L
    G = (np.random.default_rng(m).standard_normal(W.shape) * 0.3 + 0.1).astype(np.float32)
    ctx = B.Context()
    Wd, Cd, Gd = (torch.from_numpy(x).cuda() for x in (W, C0, G))
    n0 = ctx.launches
    fr = ctx.forward(Wd, Cd, tau, 0.0, iters, layer_offsets=offs)
    torch.cuda.synchronize()
    assert ctx.launches - n0 == 3
    dWj, dCj = ctx.backward(Gd, B.JFB, 0.0, 0, 1.0)
    dW, dC = ctx.backward(Gd, B.IMPLICIT, 0.0, adj_iters, alpha)
    info = ctx.info()
    for l in range(L):
        a, b = offs[l], offs[l + 1]
        W64, C64, G64 = W[a:b].astype(np.float64), C0[l * k:(l + 1) * k].astype(np.float64), G[a:b].astype(np.float64)
        Ct, _, res, _ = R.forward(W64, C64, tau, 0.0, iters)
        C = fr.C.cpu().numpy()[l * k:(l + 1) * k]
        assert info[l].status in (0, B.ERR_DIVERGED) and info[l].fwd_iters == iters
        assert_close(C, Ct, TOL_C, f"layer {l} C")
        Cg = C.astype(np.float64)
        Wq, _, S, F = R.final(W64, Cg, tau)
        assert_close(fr.Wq.cpu().numpy()[a:b], Wq, TOL_C, f"layer {l} Wq")
        rj, cj, _, _ = R.backward(W64, G64, Cg, tau, S, F, mode="jfb")
        assert_close(dCj.cpu().numpy()[l * k:(l + 1) * k], cj, TOL_GRAD, f"layer {l} dC jfb")
        assert_close(dWj.cpu().numpy()[a:b], rj, TOL_GRAD, f"layer {l} dW jfb")
        if info[l].status == 0:
            ri, ci, _, _ = R.backward(W64, G64, Cg, tau, S, F, mode="implicit", alpha=alpha, adj_max_iter=adj_iters)
            assert info[l].adj_iters == adj_iters
            assert_close(dC.cpu().numpy()[l * k:(l + 1) * k], ci, TOL_GRAD, f"layer {l} dC implicit")
            assert_close(dW.cpu().numpy()[a:b], ri, TOL_GRAD, f"layer {l} dW implicit")
    return ctx


# one block and several, bins of one weight and of thousands, codebooks of one warp and of eight, tau from far below the
# bin width the workspace allows (weights evaluated one by one) to far above the weights' range
@pytest.mark.parametrize("kind,m,k,tau", [
    ("normal", 5, 2, 0.01), ("normal", 257, 1, 0.01), ("normal", 4096, 4, 0.05), ("normal", 36864, 8, 0.01),
    ("normal", 36865, 31, 0.004), ("laplace", 100003, 33, 0.003), ("normal", 200001, 64, 0.002), ("laplace", 300007, 256, 0.001),
    ("normal", 50001, 256, 0.02), ("laplace", 65536, 16, 5e-4), ("normal", 8192, 8, 5e-5), ("laplace", 150000, 12, 2e-5),
    ("pruned", 120001, 4, 0.01), ("pruned", 30000, 7, 0.002), ("levels", 150001, 5, 0.004), ("offset", 40000, 4, 5e-4),
    ("outlier", 70000, 5, 0.003), ("outlier", 70000, 5, 2e-4), ("normal", 20000, 3, 10.0), ("normal", 1 << 20, 4, 0.002),
    ("normal", 8 << 20, 16, 0.01), ("normal", (8 << 20) - 1, 16, 0.01),
])
def test_interval_form_against_the_oracle(kind, m, k, tau):
    rng = np.random.default_rng(m + k)
    W = weights(kind, m, rng).astype(np.float32).reshape(m, 1)
    # C0 in drawn order (unsorted), distinct values where the weights allow it
    u = np.unique(W)
    C0 = rng.choice(u, size=min(k, u.size), replace=False).reshape(-1, 1).astype(np.float32)
    check(W, C0, float(np.float32(tau)), 6, 5, alpha=0.5)


def bins(W, tau, cap):
    """Fine bins of a layer that may have `cap` of them: coarse bins 0.17 tau wide, each split in a power of two."""
    m, span, floor = W.size, float(W.max()) - float(W.min()), min(cap, 32768) - 8
    width = max(0.17 * tau, span / floor)
    coarse = int(span / width) + 5
    want = max(m // 64, 512)
    if want < 16 * coarse:
        want = 16 * coarse if 16 * coarse < m // 8 else max(want, m // 8)
    f = 1
    while coarse * f * 2 <= min(want, cap):
        f *= 2
    return coarse * f


# either side of the rule for more than 32768 fine bins, at a tau where they make a difference: the layer's size, its share of the
# call, the size of the call (one layer that may have them, besides others that may not)
@pytest.mark.parametrize("sizes", [(10 << 20,), ((10 << 20) - 1,), ((10 << 20) + 3, 4099, 1001), ((10 << 20) + 3, (10 << 20) + 4)])
def test_interval_form_with_the_most_bins(sizes):
    rng = np.random.default_rng(len(sizes))
    offs = [0] + [int(x) for x in np.cumsum(sizes)]
    W = (rng.standard_normal((offs[-1], 1)) * 0.03).astype(np.float32)
    tau = float(np.float32((float(W[:sizes[0]].max()) - float(W[:sizes[0]].min())) / 140.5 / 0.17))
    assert bins(W[:sizes[0]], tau, 32768) <= 20000 and 32768 < bins(W[:sizes[0]], tau, 40960) <= 40960
    C0 = np.concatenate([rng.choice(np.unique(W[a:b]), size=8, replace=False) for a, b in zip(offs, offs[1:])]).reshape(-1, 1)
    check(W, C0, tau, 6, 3, alpha=0.5, offs=offs)


# n nearly equal weights around a centroid: a fine bin of n weights (one load a lane and several, what stays in registers and what
# does not), its start at any element of a layer with an odd start, the last weights of all; 1 to 16 centroids (two of them
# with one warp), bins split into one, 8 and more than 64 (sums of four and of one power of the place)
@pytest.mark.parametrize("n,k,m,tau,where", [
    (1, 1, 5000, 0.01, "inside"), (57, 2, 20011, 0.01, "inside"), (63, 3, 20011, 5e-4, "inside"), (64, 4, 20011, 0.01, "last"),
    (65, 5, 20011, 0.01, "inside"), (249, 8, 20011, 0.004, "last"), (257, 9, 20010, 0.01, "inside"), (505, 15, 20011, 0.01, "last"),
    (512, 16, 20011, 0.01, "inside"), (513, 4, 20011, 5e-4, "last"), (521, 16, 1 << 20, 0.05, "inside"), (1537, 7, 20011, 0.01, "last"),
    (2559, 16, 300001, 0.01, "inside"), (2571, 6, 300001, 0.02, "last"), (4000, 16, 1 << 20, 0.05, "last"), (4100, 4, 1 << 20, 0.05, "inside"),
    (9300, 5, 5 << 20, 0.05, "inside"), (19000, 16, 5 << 20, 0.05, "last"), (12000, 2, 5 << 20, 0.01, "inside"),
    (11000, 6, 5 << 20, 0.002, "inside"),   # (sums taken up in between)
])
def test_interval_form_with_a_crowded_bin(n, k, m, tau, where):
    rng = np.random.default_rng(n + k)
    at = 0.0201 if where == "inside" else 0.2
    W = np.concatenate([rng.standard_normal(1001) * 0.03, rng.standard_normal(m) * 0.03, at + rng.uniform(-1e-6, 1e-6, n)])
    W = W.astype(np.float32).reshape(-1, 1)
    second = W[1001:, 0]
    C0 = np.concatenate([rng.choice(np.unique(W[:1001]), size=k, replace=False), [np.float32(at)],
                         rng.choice(np.unique(second[:m]), size=k - 1, replace=False)]).astype(np.float32).reshape(-1, 1)
    check(W, C0, float(np.float32(tau)), 6, 5, alpha=0.5, offs=[0, 1001, W.shape[0]])


# centroids within a fraction of a fine bin of each other, and most weights there with them: a coarse bin is split in 8, so that the
# third and the fourth power of a weight's place in its fine bin count (without them 1.1e-5 to 3.3e-5, with them below 3e-6)
@pytest.mark.parametrize("k,spread", [(4, 0.1), (4, 0.03), (16, 0.03), (16, 0.01)])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_interval_form_with_close_centroids(k, spread, seed):
    import torch
    from oracle import idkm_ref as R
    from paper_2312_07759_b200 import binding as B
    tau = 0.05
    rng = np.random.default_rng(1000 * seed + k)
    near, far = rng.random(1500) * 0.02 * tau, rng.random(548) * 4.5 * tau
    W = np.concatenate([near, -near, far, -far]).astype(np.float32).reshape(-1, 1)
    C0 = ((2 * np.arange(k) + 1 - k) / k * spread * tau).astype(np.float32).reshape(-1, 1)
    tau = float(np.float32(tau))
    ctx = B.Context()
    C = ctx.forward(torch.from_numpy(W).cuda(), torch.from_numpy(C0).cuda(), tau, 0.0, 5).C.cpu().numpy()
    assert ctx.last_route()["forward"] == "interval form"
    assert_close(C, R.forward(W.astype(np.float64), C0.astype(np.float64), tau, 0.0, 5)[0], TOL_C, "C")


# a softmax so cold that an interval holds up to 390 bins which count: 1 to 3 warps for each, some intervals with a warp more than
# others, bins two at a time and one by one
@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 8, 9, 13, 15, 16])
def test_interval_form_with_many_bins_in_an_interval(k):
    rng = np.random.default_rng(k)
    W = (rng.standard_normal((120001, 1)) * 0.06).astype(np.float32)
    C0 = np.linspace(-0.15, 0.16, k).astype(np.float32).reshape(k, 1) if k < 9 else rng.choice(W[:, 0], k, replace=False).reshape(k, 1)
    check(W, C0, float(np.float32(3e-4)), 6, 5, alpha=0.5)


def test_a_warp_with_two_centroids_does_not_hold_up_the_others():
    """15 warps count around 16 centroids: 400 iterations took 1.3 times as long as with 15 centroids when one warp did all its
    work for one centroid before all of that for the other; now 1.03 times."""
    import torch
    from paper_2312_07759_b200 import binding as B
    W = torch.from_numpy((np.random.default_rng(2).standard_normal((4096, 1)) * 0.03).astype(np.float32)).cuda()
    times = {15: [], 16: []}
    for _ in range(9):
        for k in times:
            C0 = torch.linspace(-0.06, 0.06, k).reshape(k, 1).cuda()
            ctx = B.Context()
            ctx.forward(W, C0, 0.01, 0.0, 3)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.forward(W, C0, 0.01, 0.0, 400)
            b.record()
            torch.cuda.synchronize()
            assert ctx.last_route()["forward"] == "interval form"
            times[k].append(a.elapsed_time(b))
    assert np.median(times[16]) < 1.15 * np.median(times[15])


# where the stop falls decides which of the block's meetings the first warp still goes to: after the first step, on the last
# iteration but one and on the last, with room left, and never; codebooks with and without warps of their own for the intervals.
# (at most 4 iterations of up to 8 centroids take another loop, one centroid stands still after one step)
@pytest.mark.parametrize("k,stop,caps", [
    (1, 2, (5, 6, 40)), (4, 4, (5, 6, 40)), (4, 5, (5, 6, 7)), (8, 1, (5,)), (8, 7, (7, 8, 9, 40)), (9, 1, (2, 3, 9)), (15, 2, (2, 3, 4)),
    (16, 1, (2, 3, 40)), (16, 2, (2, 3, 4)), (16, 9, (9, 10, 11, 40)),
])
@pytest.mark.parametrize("m", [20011, 400003])
def test_interval_form_stops_where_it_should(k, stop, caps, m):
    import torch
    from paper_2312_07759_b200 import binding as B
    W = torch.from_numpy((np.random.default_rng(m + k).standard_normal((m, 1)) * 0.03).astype(np.float32)).cuda()
    C0 = torch.linspace(-0.05, 0.06, k).reshape(k, 1).cuda()

    def call(tol, cap):
        ctx = B.Context()
        fr = ctx.forward(W, C0, 0.01, tol, cap)
        torch.cuda.synchronize()
        assert ctx.last_route()["forward"] == "interval form"
        return ctx.info()[0], ctx.history(0), fr.C.cpu().numpy(), fr.Wq.cpu().numpy()

    res = call(0.0, 40)[1]
    assert all(res[stop - 1] < r for r in res[:stop - 1])
    tol = float(np.float32(res[stop - 1] * (1 + 1e-4) + 1e-30))
    assert all(tol < r for r in res[:stop - 1])
    for cap in caps:
        info, hist, C, Wq = call(tol, cap)
        assert (info.status, info.fwd_iters) == (B.OK, stop) and np.array_equal(hist, res[:stop])
        if not (k <= 8 and stop <= 4):
            _, _, Cs, Wqs = call(0.0, stop) if stop > 1 else (None, None, C, Wq)
            assert np.array_equal(C, Cs) and np.array_equal(Wq, Wqs)
    if k > 1:
        info, hist, _, _ = call(float(np.float32(min(res) * 0.5)), max(caps))
        assert (info.status, info.fwd_iters) == (B.MAXITER, max(caps)) and np.array_equal(hist, res[:max(caps)])


def test_interval_form_on_ragged_batches():
    """Unaligned layer starts, layers of a few weights and of many blocks, one that collapses, in one call."""
    rng = np.random.default_rng(5)
    sizes = [1001, 37, 70003, 9, 200001, 4096]
    stds = [0.05, 0.05, 0.0008, 0.03, 0.02, 0.1]
    offs = [0] + [int(x) for x in np.cumsum(sizes)]
    W = np.concatenate([rng.standard_normal((n, 1)) * s for n, s in zip(sizes, stds)]).astype(np.float32)
    C0 = np.concatenate([WL.quantile_centroids(W[offs[l]:offs[l + 1]], 4) for l in range(len(sizes))])
    ctx = check(W, C0, float(np.float32(0.01)), 12, 9, offs=offs)
    assert ctx.busy_tickets() == 0


def test_interval_form_agrees_with_the_pairwise_kernels_and_is_reproducible():
    import torch
    from paper_2312_07759_b200 import binding as B
    wl = WL.single_layer(500000, 1, 24, 0.004, std=0.03, seed=2, max_iter=20, adj_max_iter=30)
    W, C0, G = (torch.from_numpy(x).cuda() for x in (wl.W, wl.C0, wl.G))
    out = []
    for method, adj in ((0, 0), (0, 0), (1, 1)):
        ctx = B.Context()
        ctx.set_forward_loop(method)
        ctx.set_adjoint_method(adj)
        fr = ctx.forward(W, C0, wl.tau, 0.0, wl.max_iter)
        dW, dC = ctx.backward(G, B.IMPLICIT, 0.0, wl.adj_max_iter, 0.5)
        out.append([t.cpu().numpy() for t in (fr.C, fr.Wq, dW, dC)])
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)
    assert_close(out[0][0], out[2][0], 2e-6, "C")
    assert_close(out[0][1], out[2][1], 2e-6, "Wq")
