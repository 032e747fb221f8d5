"""Calls on host buffers large enough to be taken in groups of layers, against the same call as one batch (B200 only)."""
import numpy as np
import pytest

from parity_util import assert_close

pytestmark = pytest.mark.gpu


# two to four groups; a layer larger than a group's share, tiny layers between large ones, unaligned layer starts
@pytest.mark.parametrize("d,k,rows", [(1, 4, [3_000_001, 5, 3_500_003, 70_001]), (2, 4, [100_003, 2_900_001, 37, 1_700_000, 1_900_001, 12]),
                                      (4, 16, [2_000_003, 33, 3001, 1_800_001])])
def test_groups_equal_one_batch(d, k, rows):
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(d)
    offs = [0] + [int(x) for x in np.cumsum(rows)]
    W = (rng.standard_normal((offs[-1], d), dtype=np.float32) * np.float32(0.03))
    G = rng.standard_normal(W.shape, dtype=np.float32) * np.float32(0.1)
    k = min([k] + rows)
    C0 = np.concatenate([W[a:a + k] for a in offs[:-1]])
    out = []
    for one_batch in (False, True):
        ctx = B.Context()
        ctx.set_timing(one_batch)          # (phase times are of one batch)
        n0 = ctx.launches
        C, Wq, dW, dC, infos, dWj, dCj = ctx.quantize_host(W, C0, G, 0.02, 0.0, 5, B.IMPLICIT, 0.0, 6, 0.5, layer_offsets=offs, also_jfb=True)
        n = ctx.launches - n0
        assert ctx.busy_tickets() == 0 and len(infos) == len(rows)
        assert [repr(i) for i in ctx.info()] == [repr(i) for i in infos]
        out.append(([C, Wq, dW, dC, dWj, dCj], [(i.status, i.fwd_iters, i.adj_iters) for i in infos], n,
                    [ctx.history(0, l) for l in range(len(rows))]))
    assert out[0][2] > out[1][2]           # (the first call was split)
    assert out[0][1] == out[1][1]
    for name, a, b in zip(("C", "Wq", "dW", "dC", "dW jfb", "dC jfb"), out[0][0], out[1][0]):
        assert_close(a, b, 2e-5 if d > 1 else 2e-4, name, l2_only=True)
    for a, b in zip(out[0][3], out[1][3]):
        assert len(a) == len(b) == 5 and np.allclose(a, b, rtol=1e-3, atol=1e-6)


# one array for two purposes: (input, output) pairs that share their memory, one batch and several groups
@pytest.mark.parametrize("rows", [[900_001], [2_000_003, 1_900_001, 1_900_005]])
@pytest.mark.parametrize("pairs", [[("G", "Wq")], [("G", "dW"), ("W", "Wq"), ("C0", "C")], [("G", "Wq"), ("W", "dW"), ("C0", "dC")]])
def test_results_may_go_where_inputs_came_from(rows, pairs):
    import torch
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(len(rows))
    offs, d, k = [0] + [int(x) for x in np.cumsum(rows)], 2, 4
    W = rng.standard_normal((offs[-1], d), dtype=np.float32) * np.float32(0.03)
    G = rng.standard_normal(W.shape, dtype=np.float32) * np.float32(0.1)
    C0 = np.concatenate([W[a:a + k] for a in offs[:-1]])
    names = ("C", "Wq", "dW", "dC")
    got = []
    for shared in (False, True):
        pin = lambda x: torch.from_numpy(x.copy()).pin_memory().numpy()
        ins = {"W": pin(W), "G": pin(G), "C0": pin(C0)}
        out = {n: pin(np.zeros_like(W if n in ("Wq", "dW") else C0)) for n in names}
        if shared:
            out.update({o: ins[i] for i, o in pairs})
        res = B.Context().quantize_host(ins["W"], ins["C0"], ins["G"], 0.02, 0.0, 2, B.JFB, 0.0, 0, 1.0, layer_offsets=offs, out=out)
        got.append([x.copy() for x in res[:4]])
    for n, a, b in zip(names, *got):
        assert np.array_equal(a, b), n


# a large layer and a small cold one, which lands in a group of its own: quadruples with a codebook whose single layers have a
# loop of their own, and scalar weights that would be few and cold
@pytest.mark.parametrize("d,k,rows,tau", [(4, 16, [1_600_000, 2048], 5e-4), (1, 4, [6_500_001, 3000], 1e-3), (4, 64, [2_000_000, 3000, 2_000_000, 1000], 2e-3)])
def test_a_group_takes_the_routes_of_the_whole_call(d, k, rows, tau):
    """The routes are counted in launches: groups of one layer must not take what only single layers take."""
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(k)
    offs = [0] + [int(x) for x in np.cumsum(rows)]
    W = rng.standard_normal((offs[-1], d), dtype=np.float32) * np.float32(0.17)
    G = rng.standard_normal(W.shape, dtype=np.float32) * np.float32(0.1)
    C0 = np.concatenate([W[a:a + k] for a in offs[:-1]])
    iters, n, out = 12, [], []
    for one_batch in (False, True):
        ctx = B.Context()
        ctx.set_timing(one_batch)
        n0 = ctx.launches
        res = ctx.quantize_host(W, C0, G, tau, 0.0, iters, B.JFB, 0.0, 0, 1.0, layer_offsets=offs)
        n.append(ctx.launches - n0)
        out.append(res)
    groups = n[0] / n[1]
    assert groups == int(groups) and 2 <= groups <= 4
    assert [i.status for i in out[0][4]] == [i.status for i in out[1][4]]


def test_a_group_uses_the_bins_of_the_whole_call():
    """Two large layers of scalar weights, neither of which has most of the call: a group of one of them must not take the finer
    bins of a call of its own (the centroids would differ in their last bits)."""
    import torch
    from paper_2312_07759_b200 import binding as B
    rng = np.random.default_rng(4)
    rows = [(10 << 20) + 5, (10 << 20) + 3]
    offs = [0, rows[0], sum(rows)]
    W = rng.standard_normal((offs[-1], 1), dtype=np.float32) * np.float32(0.03)
    G = np.full_like(W, 0.01)
    C0 = np.concatenate([np.linspace(-0.08, 0.07, 12, dtype=np.float32)] * 2).reshape(-1, 1)
    tau = (float(W.max()) - float(W.min())) / 140.5 / 0.17
    ctx = B.Context()
    n0 = ctx.launches
    C = ctx.quantize_host(W, C0, G, tau, 0.0, 20, B.JFB, 0.0, 0, 1.0, layer_offsets=offs)[0]
    assert ctx.launches - n0 >= 8           # (two groups)
    ref = B.Context().forward(torch.from_numpy(W).cuda(), torch.from_numpy(C0).cuda(), tau, 0.0, 20, layer_offsets=offs).C
    assert np.array_equal(C, ref.cpu().numpy())
    alone = [B.Context().forward(torch.from_numpy(W[a:b]).cuda(), torch.from_numpy(C0[:12]).cuda(), tau, 0.0, 20).C for a, b in zip(offs, offs[1:])]
    assert not np.array_equal(C, torch.cat(alone).cpu().numpy())
