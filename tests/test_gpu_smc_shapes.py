"""The one-call filter against ppl_smc_step, particle for particle, at the sizes
where its kernels change over (one cluster of up to 16 blocks of 1024 or 2048
particles, then grid barriers) and on weights that concentrate on few
particles, whose offspring run over many slots, rows and blocks."""
import numpy as np
import pytest

import synth
from gpu_util import load_ppl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppl():
    return load_ppl()


def _stepwise(ppl, model, y, N, seed):
    import torch
    x, lw = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda")
    acc = torch.zeros(1, dtype=torch.float64, device="cuda")
    flags = torch.zeros(len(y), dtype=torch.int32, device="cuda")
    est = torch.zeros((len(y), 2), dtype=torch.float64, device="cuda")
    ws = ppl.workspace(model, N)
    for t in range(1, len(y) + 1):
        ppl.ppl_smc_step(model, float(y[t - 1]), t, seed, x, lw, acc, flags[t - 1:t], est[t - 1], ws)
    assert ppl.ppl_workspace_status(ws) == 0
    return x, lw, flags, est


# obs_sigma 0.5: the benchmark's model; 0.02 and 0.002: a step's weight lies on
# tens or a few particles (at 200000, more outputs than a block's table holds)
@pytest.mark.parametrize("sigma", [0.5, 0.02, 0.002])
@pytest.mark.parametrize("N", [2, 1023, 1024, 1025, 10000, 16384, 16385, 32768, 32769, 200000])
def test_filter_matches_stepwise(ppl, N, sigma):
    import torch
    T = 12
    model = ppl.lgssm_model(obs_sigma=sigma)
    y = synth.lgssm_dataset(T, 5)
    out = ppl.ppl_smc_run(model, torch.from_numpy(y).cuda(), N, 3)
    assert ppl.ppl_workspace_status(out["ws"]) == 0
    x, lw, flags, est = _stepwise(ppl, model, y, N, 3)
    assert torch.equal(out["resampled"], flags)
    assert torch.equal(out["x"], x)
    assert torch.equal(out["lw"], lw)
    np.testing.assert_allclose(out["ess"].cpu().numpy(), est[:, 1].cpu().numpy(), rtol=1e-5)
    assert abs(float(out["log_z"].item()) - float(est[-1, 0])) < 1e-6 * max(T, abs(float(est[-1, 0])))


@pytest.mark.parametrize("N", [3000, 50000])
def test_filter_reports_nan_and_recovers(ppl, N):
    import torch
    model = ppl.lgssm_model()
    y = torch.from_numpy(synth.lgssm_dataset(6, 5)).cuda()
    bad = y.clone()
    bad[3] = float("nan")
    out = ppl.ppl_smc_run(model, bad, N, 3)
    assert ppl.ppl_workspace_status(out["ws"]) == ppl.PPL_ENAN
    out = ppl.ppl_smc_run(model, y, N, 3, ws=out["ws"])
    assert ppl.ppl_workspace_status(out["ws"]) == 0
    # captured in a graph, the call gives the same bits
    ref = out["x"].clone()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        ppl.ppl_smc_run(model, y, N, 3, ws=out["ws"], out={k: out[k] for k in ("x", "lw", "log_z", "resampled", "ess")})
    out["x"].zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out["x"], ref)
