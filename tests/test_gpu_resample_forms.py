"""The resampler's scatter form (row marks) at the edges of its rows, records
and plans."""
import numpy as np
import pytest

import synth
from gpu_util import load_ppl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppl():
    return load_ppl()


# A shard's plan says where its outputs lie; one that its weights do not bear out
# is refused and writes nothing (the buffers hold room for what it claims).
@pytest.mark.parametrize("change", ["none", "k_end+1", "k_end-1", "k_first+1", "k_first-1", "c_base",
                                    "stride", "offset", "weights"])
@pytest.mark.parametrize("N,M", [(40000, 40000), (5000, 1 << 20)])
def test_plan_that_does_not_fit_the_weights(ppl, N, M, change):
    import torch
    lw = torch.from_numpy(synth.log_weights(N, 9, "normal", scale=1.0)).cuda()
    h = N // 2 + 77
    mx = lw.max().double().reshape(1)
    shards = [lw[:h].clone(), lw[h:].clone()]
    totals = [int(ppl.ppl_resample_shard_total(s, mx, N).item()) for s in shards]
    plan = ppl.ppl_resample_shard_plan(np.array(totals, dtype=np.uint64), N, M, 3)[1]
    n_out = plan.k_end - plan.k_first
    anc = torch.full((n_out + 512,), -7, dtype=torch.int32, device="cuda")
    rec = torch.arange(8 * (N - h), dtype=torch.float32, device="cuda").view(N - h, 8)
    out = torch.full((n_out + 512, 8), -7.0, device="cuda")
    if change == "k_end+1":
        plan.k_end, plan.m = plan.k_end + 1, plan.m + 1
    elif change == "k_end-1":
        plan.k_end -= 1
    elif change == "k_first+1":
        plan.k_first += 1
    elif change == "k_first-1":
        plan.k_first -= 1
    elif change == "c_base":
        plan.c_base += 2 * plan.stride
    elif change == "stride":
        plan.stride += plan.stride // 2
    elif change == "offset":
        plan.offset = plan.stride
    elif change == "weights":
        shards[1][100] -= 5.0
        shards[1][1000:1100] -= 1.0
    ws = ppl.workspace(ppl.poly_model(), N)
    ppl.ppl_resample_shard(shards[1], h, mx, plan, ancestors=anc, state_in=rec, state_out=out, ws=ws)
    if change == "none":
        assert ppl.ppl_workspace_status(ws) == 0
        assert torch.equal(out[:n_out], rec[anc[:n_out].long() - h])
    else:
        assert ppl.ppl_workspace_status(ws) == ppl.PPL_EINVAL
        assert bool((anc == -7).all()) and bool((out == -7.0).all())
    assert bool((anc[n_out:] == -7).all()) and bool((out[n_out:] == -7.0).all())


def _gather_check(ppl, orc, lw, M, state, seed=13):
    import torch
    st, ref = orc.resample_from_lw(lw, M, seed, 1, 3)
    assert st == 0
    anc, out = ppl.ppl_resample_gather(M, seed, torch.from_numpy(lw).cuda(), state, instance=1, t=3)
    assert np.array_equal(anc.cpu().numpy(), ref)
    assert torch.equal(out.view(torch.uint8), state[anc.long()].view(torch.uint8))


# Runs of one particle's offspring over none, one, several and all rows of its
# chunk, several long runs at once, and up to the most outputs that a chunk
# writes in this form (8192).
@pytest.mark.parametrize("M", [33, 4096, 7001, 8192, 8193, 20000])
@pytest.mark.parametrize("N", [1, 40, 4096, 10000])
def test_runs_over_many_rows(ppl, orc, N, M):
    import torch
    rng = np.random.default_rng([N, M])
    state = torch.from_numpy(rng.standard_normal((N, 6)).astype(np.float32)).cuda()
    for scale in (0.5, 4.0, 10.0, 40.0):
        _gather_check(ppl, orc, (scale * rng.standard_normal(N)).astype(np.float32), M, state)
    lw = np.full(N, -np.inf, dtype=np.float32)
    lw[N // 2] = 0.0  # one particle takes everything
    _gather_check(ppl, orc, lw, M, state)
    lw[:] = -1.25     # all alike: runs of M / N
    _gather_check(ppl, orc, lw, M, state)


# Records of every kind the fused gather distinguishes: 4-byte words past one
# round of a row's copies, the widest record, 32-byte records that lie 4 or 16
# bytes off a 32-byte boundary; near-uniform and concentrated weights, rows and
# chunks that end ragged.
@pytest.mark.parametrize("words,shift", [(5, 0), (6, 0), (7, 0), (255, 0), (256, 0), (8, 1), (8, 4),
                                         (12, 0), (12, 2), (4, 4)])
@pytest.mark.parametrize("N,M", [(4099, 4099), (9000, 17999), (5000, 4097)])
def test_record_kinds(ppl, orc, words, shift, N, M):
    import torch
    rng = np.random.default_rng([N, words])
    def room(n):
        return torch.empty(n * words + shift, device="cuda")[shift:].view(n, words)
    state, out = room(N), room(M)
    state.copy_(torch.from_numpy(rng.standard_normal((N, words)).astype(np.float32)))
    for lw in (np.full(N, -1.25, dtype=np.float32), synth.log_weights(N, 5, "normal", scale=0.3),
               synth.log_weights(N, 6, "normal", scale=12.0)):
        st, ref = orc.resample_from_lw(lw, M, 13, 1, 3)
        assert st == 0
        anc, got = ppl.ppl_resample_gather(M, 13, torch.from_numpy(lw).cuda(), state, state_out=out,
                                           instance=1, t=3)
        assert np.array_equal(anc.cpu().numpy(), ref)
        assert got.data_ptr() == out.data_ptr() and torch.equal(out, state[anc.long()])


@pytest.mark.parametrize("words", [6, 12])
def test_sharded_gather_of_other_records(ppl, words):
    import torch
    N, M = 30011, 30011
    lw = torch.from_numpy(synth.log_weights(N, 9, "normal", scale=1.0)).cuda()
    state = torch.randn(N, words, device="cuda")
    anc_ref, rec_ref = ppl.ppl_resample_gather(M, 3, lw, state)
    b = [0, 11000, 11001, N]
    mx = lw.max().double().reshape(1)
    parts = [lw[b[g]:b[g + 1]].clone() for g in range(3)]
    totals = [int(ppl.ppl_resample_shard_total(p, mx, N).item()) for p in parts]
    plans = ppl.ppl_resample_shard_plan(np.array(totals, dtype=np.uint64), N, M, 3)
    got = [ppl.ppl_resample_shard(parts[g], b[g], mx, plans[g],
                                  state_in=state[b[g]:b[g + 1]].clone()) for g in range(3)]
    assert torch.equal(torch.cat([g[0] for g in got]), anc_ref)
    assert torch.equal(torch.cat([g[1] for g in got]), rec_ref)


def test_most_outputs_with_a_stride_of_one(ppl):
    # the most outputs there are, fixed-point weights whose sum is just below twice
    # their number: stride 1, and the last chunk's sums lie almost 2^31 positions
    # past its last output
    import torch
    M = (1 << 31) - 1
    q = torch.ones(2 * 4096, dtype=torch.int64)
    q[0] = M - 100 - 4095   # chunk 0: the first M - 100 positions
    q[4096:] = 0
    q[4096], q[4097], q[5000] = 40, 30, 7
    q[6000], q[6001] = 100, M - 100 - 30 - 40 - 7 - 100 + 99 + 100
    total = int(q.sum())
    assert M <= total < 2 * M
    anc = ppl.ppl_resample(M, 5, q_fixed=q.cuda())
    c = torch.cumsum(q.cuda(), 0)
    for k in range(0, M, 1 << 28):  # output k's position is k: the first sum above it
        pos = torch.arange(k, min(k + (1 << 28), M), device="cuda")
        assert torch.equal(anc[k:k + len(pos)].long(), torch.searchsorted(c, pos, right=True))
