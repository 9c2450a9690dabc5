"""Joint test on the CUDA cores (fp32 caches, 64-channel heads) against the
oracle's scan, at the sizes where its staging changes: rounds whose pages fit
the 64-row chunk buffers together, rounds that exceed them, pages longer than
a chunk, ragged row groups, and more row groups than resident blocks.  The
bound is the effect tolerance of the cache's type, up to the first decision
that lies within it."""
import numpy as np
import pytest
import torch

from oracle import core
from oracle_bridge import OracleStep, isclose_tol, rel_close, safe_threshold_mask
from paper_2608_07855_gb300 import commitkv as ck
from paper_2608_07855_gb300 import synth
from paper_2608_07855_gb300.workload import DeviceTrajectory, StepBuffers

pytestmark = pytest.mark.gpu

CONFIGS = [dict(G=8), dict(G=16, d=128), dict(G=24, dtype="bf16"), dict(G=100, L_pre=900, L_obs=80, B=400),
           dict(G=16, W=3), dict(G=16, M=6, H=8, Hq=16, W=64, L_pre=300, L_obs=40, B=128)]


@pytest.mark.parametrize("kw", CONFIGS, ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items()))
def test_joint_steps_and_decisions(kw):
    base = dict(dtype="f32", d=64, H=2, Hq=4, M=1, W=16, L_pre=500, L_obs=60, B=200, outlier_channels=0)
    cfg = synth.small_config("cores", **dict(base, **kw))
    tr = synth.make_trajectory(cfg, 5)
    o = OracleStep(tr, "explicit")
    dev = DeviceTrajectory.upload(tr)
    b = StepBuffers(cfg, [dev])
    Rp = o.R_post
    pages = [E for E in np.argsort(Rp, kind="stable") if np.isfinite(Rp[E]) and Rp[E] > 0][:15]
    cand_np = np.array(pages, np.int64)[np.random.default_rng(5).permutation(len(pages))]
    nc = len(cand_np)
    tau = float(np.float32(np.quantile(Rp[cand_np], 0.5)))
    acc_o, step_o = core.greedy(o.post, cand_np, tau, "closed", stats=o.stats)
    b.score_post()
    cand = torch.zeros(dev.P_post, dtype=torch.int32, device="cuda")
    cand[:nc] = torch.from_numpy(cand_np.astype(np.int32)).cuda()
    n_cand = torch.tensor([nc], dtype=torch.int32, device="cuda")
    ck.commitkv_joint_test(b.shape, [dev.post()], b.stats, [cand], n_cand, tau, b.accepted, b.step_R, workspace=b.ws)
    assert b.status() == ck.COMMITKV_OK
    step = b.step_R[0].cpu().numpy()[:nc]
    acc = b.accepted[0].cpu().numpy()[:dev.P_post]
    tol = isclose_tol(cfg.dtype)
    safe = safe_threshold_mask(step_o, tau, tol)
    upto = nc if safe.all() else int(np.argmin(safe)) + 1
    assert rel_close(step[:upto], step_o[:upto], tol).all(), (step[:upto], step_o[:upto])
    assert np.array_equal(acc[cand_np[:upto - 1]], acc_o[cand_np[:upto - 1]])
    assert np.array_equal(acc[cand_np] != 0, step <= tau)
    assert acc.sum() == (step <= tau).sum()
