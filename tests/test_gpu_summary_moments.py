"""Second moments of the posterior summary where the FP32 sums behind them are
hardest to combine, against FP64."""
import numpy as np
import pytest

import synth
from gpu_util import load_ppl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppl():
    return load_ppl()


def _records(n, c):
    rec = np.zeros((len(n), 8), dtype=np.float32)
    rec[:, :6] = c
    rec[:, 6] = n.astype(np.int32).view(np.float32)
    return rec


def _reduce(ppl, n, c, lw):
    import torch
    return ppl.read_result(ppl.ppl_posterior_reduce(
        ppl.poly_model(), torch.from_numpy(_records(n, c)).cuda(), torch.from_numpy(lw).cuda()))


# The tiles of 128 particles go round the blocks (one per SM): block 0 holds
# nothing but each degree's best trace, `dist` standard deviations from the
# others, which sets the point the final merge works around.  What a block
# passes on is FP32 (about 1e-6 of its own variance); the merge must not add to
# it, whatever the distance.
@pytest.mark.parametrize("dist", [0.0, 10.0, 100.0, 1000.0])
def test_best_trace_alone_in_its_block(ppl, orc, dist):
    import torch
    blocks = torch.cuda.get_device_properties(0).multi_processor_count
    N = blocks * 128 * 64
    rng = np.random.default_rng(17)
    n = rng.integers(2, 6, N)
    c = rng.standard_normal((N, 6)).astype(np.float32)
    lw = rng.uniform(-1.5, -0.5, N).astype(np.float32)
    lw[(np.arange(N) // 128) % blocks == 0] = -np.inf
    for d in range(4):
        i = 7 + 30 * d
        n[i], lw[i], c[i] = 2 + d, 0.0, dist
    c[np.arange(6)[None, :] > n[:, None]] = 0
    out = _reduce(ppl, n, c, lw)
    ref = orc.posterior_poly(orc.poly_model(), lw.astype(np.float64), n.astype(np.int32),
                             c.astype(np.float64))
    assert out["status"] == 0 and list(out["deg_argmax"]) == [7, 37, 67, 97]
    for d in range(4):
        live = slice(0, d + 3)
        var = ref["deg_var"][d][live]
        assert np.all(np.abs(out["deg_var"][d][live] - var) <= 1e-5 * var), (d, out["deg_var"][d], var)
        err = np.abs(out["deg_mean"][d][live] - ref["deg_mean"][d][live])
        assert np.all(err <= 1e-6 * (np.sqrt(var) + np.abs(ref["deg_mean"][d][live])))


# One coefficient whose square leaves FP32's range: with a weight that FP32
# rounds to 0, or one that makes it the whole variance of its own degree; in the
# midst of others, and as the first of its degree that its warp meets (where it
# sets the point that the warp's sums are taken around).
@pytest.mark.parametrize("first", [False, True])
@pytest.mark.parametrize("lw_far", [-300.0, -69.0])
def test_coefficient_whose_square_overflows(ppl, orc, lw_far, first):
    N, at = 40000, 5
    rng = np.random.default_rng(3)
    n = rng.integers(2, 6, N)
    c = rng.standard_normal((N, 6)).astype(np.float32)
    lw = rng.uniform(-1.5, 0.0, N).astype(np.float32)
    n[:128] = 3
    if first:
        n[:128] = np.where(np.arange(128) % 2 == 0, 2, 4)
    n[at] = 3
    c[np.arange(6)[None, :] > n[:, None]] = 0
    c[at, 1] = 1e20
    lw[at] = lw_far
    out = _reduce(ppl, n, c, lw)
    ref = orc.posterior_poly(orc.poly_model(), lw.astype(np.float64), n.astype(np.int32),
                             c.astype(np.float64))
    assert out["status"] == 0
    for d in range(4):
        live = slice(0, d + 3)
        var = ref["deg_var"][d][live]
        assert np.all(np.abs(out["deg_var"][d][live] - var) <= 1e-5 * var), (d, out["deg_var"][d], var)


# A moment that FP32 cannot hold is reported as such: a NaN coefficient that
# carries weight shows in its variance as in its mean, and one of 1e20
# with an ordinary weight gives no finite variance.
@pytest.mark.parametrize("N", [100, 5000])
@pytest.mark.parametrize("value", [float("nan"), 1e20])
def test_moments_out_of_range_are_not_hidden(ppl, value, N):
    rng = np.random.default_rng(4)
    n = np.full(N, 3)
    c = rng.standard_normal((N, 6)).astype(np.float32)
    c[:, 4:] = 0
    c[N // 2, 1] = value
    out = _reduce(ppl, n, c, np.zeros(N, dtype=np.float32))
    assert not np.isfinite(out["deg_var"][1][1])
    assert np.isnan(out["deg_mean"][1][1]) == np.isnan(value)
    assert np.all(np.isfinite(out["deg_var"][1][[0, 2, 3]]))


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_nan_traces_of_one_degree_leave_the_others(ppl, value):
    # a proposal whose third degree holds a NaN mean (or an infinite one), in a batch large enough for the
    # kernel that keeps lane sums: the status tells, and the other degrees'
    # moments are those of the same proposal without it, bit for bit
    import torch
    sets, N = 4, 1 << 23
    d = synth.prior_datasets(sets, 16, 5)
    doff, poff = np.arange(sets + 1) * 16, np.arange(sets + 1) * N
    model = ppl.poly_model()
    ws = ppl.batched_workspace(doff, poff)
    plan = ppl.ppl_batched_prepare(model, doff, poff, 8, 2, ws)
    x, y = (torch.from_numpy(np.ascontiguousarray(d[k], dtype=np.float32).reshape(-1)).cuda() for k in "xy")
    do, po = torch.from_numpy(doff).cuda(), torch.from_numpy(poff).cuda()
    prop = torch.zeros((sets, 48), device="cuda")
    rows = []
    for bad in (False, True):
        if bad:
            prop[1, 4 + 2 * 7] = value  # degrees 2 and 3 take 3 + 4 slots
        out = ppl.batch_results_tensor(sets)
        ppl.ppl_infer_is_learned(model, x, y, do, po, 7, plan, prop, out, ws)
        assert ppl.ppl_batched_status(ws) == (ppl.PPL_ENAN if bad else 0)
        rows.append(ppl.read_batch_results(out, sets))
    good, bad = rows
    for f in ("deg_mean", "deg_var", "deg_argmax"):
        assert np.array_equal(good[0][f], bad[0][f]) and np.array_equal(good[3][f], bad[3][f])
        others = [0, 1, 3]
        assert np.array_equal(np.asarray(good[1][f])[others], np.asarray(bad[1][f])[others]), f
    assert bad[1]["deg_argmax"][2] == -1 and bad[1]["p_n"][2] == 0.0
