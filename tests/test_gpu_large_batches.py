"""Large batches of short data sets (the kernel of lane sums) under proposals of
their own, against the oracle and against the kernel of smaller batches."""
import numpy as np
import pytest

import oracle.mlp as mlp
import synth
from gpu_util import check_summary, load_ppl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppl():
    return load_ppl()


def _run(ppl, d, prop, N, ppt, seed):
    import torch
    B = len(N)
    doff, poff = np.arange(B + 1) * 32, np.concatenate([[0], np.cumsum(N)])
    model = ppl.poly_model()
    ws = ppl.batched_workspace(doff, poff)
    plan = ppl.ppl_batched_prepare(model, doff, poff, ppt, 2, ws)
    t = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in
         (d["x"][:B].reshape(-1), d["y"][:B].reshape(-1), doff, poff, prop[:B])]
    out = ppl.batch_results_tensor(B)
    ppl.ppl_infer_is_learned(model, t[0], t[1], t[2], t[3], seed, plan, t[4], out, ws)
    assert ppl.ppl_batched_status(ws) == 0
    return ppl.read_batch_results(out, B)


# Every instance has its own proposal and data, and sizes around the runs of
# 16384 traces, so that a block's run ends in one instance and goes on in the
# next: a proposal or data set left over from the last one would show.  The
# larger instances come last: without them the batch is below the kernel's
# limit, and the instances before them run in the kernel of smaller batches with
# the same draws.
@pytest.mark.parametrize("ppt", [2, 8])
def test_learned_proposals_across_runs(ppl, orc, ppt):
    W = synth.mlp_weights(11, bias_scale=0.3)
    sizes = [16383, 16385, 1, 30011, 12000, 16384, 50021, 700, 20000]
    big = [1 << 23, (1 << 23) + 5, 1 << 23, 1 << 23]
    n = len(sizes)
    d = synth.prior_datasets(n + len(big), 32, 12)
    prop = np.stack([mlp.forward(W, mlp.features(d["x"][b], d["y"][b]))[0]
                     for b in range(n + len(big))]).astype(np.float32)
    # (each instance's degree logits and spreads its own, so that no two agree)
    prop[:, :4] += np.random.default_rng(5).normal(0, 0.7, (n + len(big), 4)).astype(np.float32)
    large = _run(ppl, d, prop, np.array(sizes + big, dtype=np.int64), ppt, 6)
    small = _run(ppl, d, prop, np.array(sizes + [1000] * len(big), dtype=np.int64), ppt, 6)
    m = orc.poly_model()
    for b in range(n):
        lw, deg, c = mlp.learned_is(m, prop[b].astype(np.float64), d["x"][b], d["y"][b], sizes[b], 6,
                                    instance=b)
        ref = orc.posterior_poly(m, lw, deg, c)
        for r in (large[b], small[b]):
            assert r["status"] == 0
            assert abs(r["log_z"] - ref["log_z"]) <= 1e-3 + 2.0 ** -21 * abs(ref["max_lw"]), b
            assert r["ess"] == pytest.approx(ref["ess"], rel=1e-3), b
            check_summary(r, ref, b)
        # the same draws and log-weights in both kernels; the sums differ in order
        assert large[b]["max_lw"] == small[b]["max_lw"] and large[b]["argmax"] == small[b]["argmax"]
        assert np.array_equal(large[b]["deg_argmax"], small[b]["deg_argmax"])
        assert large[b]["log_z"] == pytest.approx(small[b]["log_z"], abs=1e-5), b
        assert large[b]["ess"] == pytest.approx(small[b]["ess"], rel=1e-5), b
        np.testing.assert_allclose(large[b]["p_n"], small[b]["p_n"], rtol=1e-5)
    for b in range(n, n + len(big)):
        assert large[b]["status"] == 0 and large[b]["n_particles"] == big[b - n]
        assert np.isfinite(large[b]["log_z"]) and large[b]["ess"] > 0


def test_autotuner_times_one_number_of_blocks(ppl, tmp_path):
    # the kernel of large batches has its own number of blocks: the candidates that
    # differ in nothing else are one launch, timed once
    import torch
    B, N = 64, 1 << 19
    d = synth.prior_datasets(B, 16, 3)
    doff, poff = np.arange(B + 1) * 16, np.arange(B + 1) * N
    t = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in
         (d["x"].astype(np.float32).reshape(-1), d["y"].astype(np.float32).reshape(-1), doff, poff)]
    model = ppl.poly_model()
    ws = ppl.batched_workspace(doff, poff)
    out = ppl.batch_results_tensor(B)
    for k in range(4):
        plan = ppl.ppl_batched_autotune(model, *t, doff, poff, k, out, ws,
                                        str(tmp_path / f"tune{k}.json"))
        assert plan.blocks_per_sm == 2
