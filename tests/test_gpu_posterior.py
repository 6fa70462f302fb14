"""The posterior summary of given populations against the oracle at the edges
of the kernel's warp tiles (128 particles, 16 warps a block) and on weights
that move its reference point in every way."""
import numpy as np
import pytest

from gpu_util import check_summary, load_ppl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppl():
    return load_ppl()


def _population(N, kind, rng):
    n = rng.integers(2, 6, N).astype(np.int32)
    c = rng.normal(0, 3, (N, 6)).astype(np.float32)
    lw = rng.normal(-30, 4, N).astype(np.float32)
    if kind == "rising":      # every particle the best so far: the reference keeps moving
        lw = np.linspace(-900, -1, N).astype(np.float32)
    elif kind == "onehot":
        lw = np.full(N, -np.inf, dtype=np.float32)
        lw[N // 2] = -3.0
    elif kind == "narrow":    # moments far from 0 next to their spread
        c = (50 + 0.01 * rng.standard_normal((N, 6))).astype(np.float32)
    elif kind == "one_degree":
        n[:] = 4
    c[np.arange(6)[None, :] > n[:, None]] = 0
    return n, c, lw


@pytest.mark.parametrize("kind", ["normal", "rising", "onehot", "narrow", "one_degree"])
@pytest.mark.parametrize("N,shift", [(1, 0), (127, 1), (129, 0), (2049, 3), (311299, 1), (1 << 20, 0)])
def test_posterior_reduce_edges(ppl, orc, N, shift, kind):
    import torch
    n, c, lw = _population(N, kind, np.random.default_rng([N, len(kind)]))
    rec = np.zeros((N, 8), dtype=np.float32)
    rec[:, :6] = c
    rec[:, 6] = n.view(np.float32)
    # log-weights off a 16-byte boundary by `shift` floats, records 16 bytes
    # off a 32-byte one when shift is odd
    lw_d = torch.empty(N + shift, device="cuda")[shift:]
    lw_d.copy_(torch.from_numpy(lw))
    buf = torch.empty(8 * N + 4, device="cuda")
    rec_d = buf[4 * (shift & 1):][:8 * N].view(N, 8)
    rec_d.copy_(torch.from_numpy(rec))
    out = ppl.read_result(ppl.ppl_posterior_reduce(ppl.poly_model(), rec_d, lw_d))
    ref = orc.posterior_poly(orc.poly_model(), lw.astype(np.float64), n, c.astype(np.float64))
    assert out["status"] == 0 and out["argmax"] == ref["argmax"]
    assert np.array_equal(out["deg_argmax"], ref["deg_argmax"])
    assert out["log_z"] == pytest.approx(ref["log_z"], abs=1e-6 * max(1.0, abs(ref["log_z"])))
    assert out["ess"] == pytest.approx(ref["ess"], rel=1e-5)
    check_summary(out, ref, (N, kind))


def test_posterior_reduce_reports_bad_records(ppl):
    import torch
    N = 3000
    rec = torch.zeros(N, 8, device="cuda")
    rec[:, 6] = torch.full((N,), 3, dtype=torch.int32, device="cuda").view(torch.float32)
    rec[2999, 6] = torch.tensor([17], dtype=torch.int32, device="cuda").view(torch.float32)[0]
    rec[2999, :6] = float("nan")  # the record of no degree is left out whole
    ws = ppl.workspace(ppl.poly_model(), N)
    out = ppl.read_result(ppl.ppl_posterior_reduce(ppl.poly_model(), rec, None, ws=ws))
    assert ppl.ppl_workspace_status(ws) == ppl.PPL_EINVAL
    assert out["p_n"][1] == 1.0 and np.all(np.isfinite(out["deg_mean"]))
    lw = torch.zeros(N, device="cuda")
    lw[5] = float("nan")
    rec[2999] = rec[0]
    ppl.ppl_posterior_reduce(ppl.poly_model(), rec, lw, ws=ws)
    assert ppl.ppl_workspace_status(ws) == ppl.PPL_ENAN
