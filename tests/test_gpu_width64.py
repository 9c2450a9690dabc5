"""Tensor-core scoring of 64-channel bf16 heads against the fp64 oracle.  P is
carried as three bf16 terms (2^-25), so the bounds are those of the fp32
kernels: 1e-4 on the effects, 1e-5 on the row statistics."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_07855_gb300 import commitkv as ck
from paper_2608_07855_gb300 import synth
from paper_2608_07855_gb300.workload import DeviceTrajectory, StepBuffers

pytestmark = pytest.mark.gpu

# a row tile and two with a ragged end; pages shorter and longer than a slot
# and a tile; a cache shorter than a tile
CONFIGS = [dict(), dict(W=40, G=16, L_pre=600, L_obs=70, B=256), dict(G=100, L_pre=900, L_obs=80, B=400),
           dict(G=200, H=4, Hq=4, W=8, L_pre=1500, L_obs=300), dict(W=4, G=8, L_pre=60, L_obs=20, B=16, planted_frac=0.0,
                                                                    event_len=(8, 20))]


@pytest.mark.parametrize("kw", CONFIGS, ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items()) or "base")
def test_effects_and_stats_of_64_channel_heads(kw):
    cfg = synth.small_config("w64", **dict(dict(d=64, plant="shared", alpha=4.0, beta=(2.0, 3.0), gamma=4.0), **kw))
    tr = synth.make_trajectory(cfg, 3)
    dev = DeviceTrajectory.upload(tr)
    buf = StepBuffers(cfg, [dev])
    head = [torch.zeros(cfg.M, cfg.Hq, dev.P_post, device="cuda")]
    buf.score()
    Rp = torch.zeros(dev.P_post, device="cuda")
    ck.commitkv_page_effects(buf.shape, [dev.post()], [Rp], head_R_out=head, workspace=buf.ws)
    assert buf.status() == ck.COMMITKV_OK
    # the same call without maxima per head, in one batch with the pre-commit cache, which
    # both take the tensor cores; with statistics the post-commit cache took the CUDA cores
    Rq = [torch.zeros(tr.P_pre, device="cuda"), torch.zeros(dev.P_post, device="cuda")]
    ck.commitkv_page_effects(buf.shape, [dev.pre(), dev.post()], Rq, workspace=buf.ws)
    assert buf.status() == ck.COMMITKV_OK
    assert torch.equal(Rq[1], Rp) and torch.equal(Rq[0], buf.R_pre[0][:tr.P_pre])

    def f64(a):
        return synth.values_f64(a, "bf16")

    L = tr.L_pre
    pre = oracle.Problem(f64(tr.K)[:, :, :L], f64(tr.V)[:, :, :L], tr.pos[:L], f64(tr.Q_pre), tr.qpos_pre,
                         tr.page_start[:tr.P_pre], tr.page_len[:tr.P_pre])
    post = oracle.Problem(f64(tr.K), f64(tr.V), tr.pos, f64(tr.Q_post), tr.qpos_post, tr.page_start, tr.page_len)
    for got, prob, per_head in ((Rq[0], pre, None), (Rp, post, head[0]), (buf.R_post[0], post, None)):
        want = oracle.page_effects(prob, "closed")
        for g, w in ((got, want[0]), (per_head, want[1])):
            if g is None:
                continue
            g = g.cpu().numpy().reshape(-1)
            w = np.asarray(w).reshape(-1)
            fin = np.isfinite(w)
            assert np.array_equal(np.isfinite(g), fin)
            assert np.all(np.abs(g[fin] - w[fin]) <= 1e-4 * np.abs(w[fin]) + 1e-30)
    m, l, o, n = oracle.row_stats(post)
    st = buf.stats[0].cpu().numpy().reshape(-1, cfg.d + 4)
    assert np.array_equal(st[:, 2].astype(np.int64), n)
    assert np.all(np.abs(st[:, 0] - m) <= 1e-5 * np.abs(m) + 1e-6)
    assert np.all(np.abs(st[:, 1] - l) <= 1e-5 * l)
    assert np.all(np.linalg.norm(st[:, 4:] - o, axis=1) <= 1e-5 * np.linalg.norm(o, axis=1))
    # the page pass alone, from the exact statistics
    exact = np.concatenate([np.stack([m, l, n], 1), np.zeros((len(m), 1)), o], 1).astype(np.float32)
    R2 = torch.zeros_like(Rp)
    ck.commitkv_page_effects_from_stats(buf.shape, [dev.post()], [torch.from_numpy(exact).cuda().view_as(buf.stats[0])], [R2],
                                        workspace=buf.ws)
    assert buf.status() == ck.COMMITKV_OK
    w = np.asarray(oracle.page_effects(post, "closed")[0])
    fin = np.isfinite(w) & (w > 0)
    g = R2.cpu().numpy().astype(np.float64)
    assert np.array_equal(np.isfinite(g), np.isfinite(w))
    assert np.linalg.norm(g[fin] - w[fin]) <= 1e-5 * np.linalg.norm(w[fin])
    # from the call's own statistics: the effects of that call
    ck.commitkv_page_effects_from_stats(buf.shape, [dev.post()], [buf.stats[0]], [R2], workspace=buf.ws)
    assert buf.status() == ck.COMMITKV_OK
    assert torch.equal(R2, buf.R_post[0])
