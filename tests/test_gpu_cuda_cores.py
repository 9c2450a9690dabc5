"""Scoring on the CUDA cores (fp32 caches) against the fp64 oracle at the
sizes where its work is split: caches of one chunk (128 tokens) less, exactly
and more, pages that cross the 64-token windows and that are longer than one,
row groups with a ragged end, and a value row of infinities.  The bounds are
those of fp32 inputs: 1e-4 on the effects, 1e-5 on the row statistics."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_07855_gb300 import commitkv as ck
from paper_2608_07855_gb300 import synth
from paper_2608_07855_gb300.workload import DeviceTrajectory, StepBuffers

pytestmark = pytest.mark.gpu

CONFIGS = [dict(L_pre=107), dict(L_pre=108), dict(L_pre=109, d=128), dict(W=33, G=24), dict(G=100, W=5, d=128),
           dict(W=3, G=7, L_pre=700)]


def _case(kw):
    base = dict(dtype="f32", d=64, H=2, Hq=4, M=1, W=16, G=16, L_pre=500, L_obs=20, B=64, outlier_channels=0,
                plant="shared", alpha=4.0, beta=(2.0, 3.0), gamma=4.0, event_len=(8, 20))
    cfg = synth.small_config("cuda_cores", **dict(base, **kw))
    return cfg, synth.make_trajectory(cfg, 7)


@pytest.mark.parametrize("kw", CONFIGS, ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items()))
def test_effects_and_stats(kw):
    cfg, tr = _case(kw)
    dev = DeviceTrajectory.upload(tr)
    buf = StepBuffers(cfg, [dev])
    head = [torch.zeros(cfg.M, cfg.Hq, dev.P_post, device="cuda")]
    buf.score()
    Rp = torch.zeros(dev.P_post, device="cuda")
    ck.commitkv_page_effects(buf.shape, [dev.post()], [Rp], head_R_out=head, workspace=buf.ws)
    assert buf.status() == ck.COMMITKV_OK
    assert torch.equal(Rp, buf.R_post[0])
    post = oracle.Problem(np.asarray(tr.K, np.float64), np.asarray(tr.V, np.float64), tr.pos,
                          np.asarray(tr.Q_post, np.float64), tr.qpos_post, tr.page_start, tr.page_len)
    R, per_head = oracle.page_effects(post, "closed")[:2]
    for g, w in ((Rp, R), (head[0], per_head)):
        g, w = g.cpu().numpy().reshape(-1), np.asarray(w).reshape(-1)
        fin = np.isfinite(w)
        assert np.array_equal(np.isfinite(g), fin)
        assert np.all(np.abs(g[fin] - w[fin]) <= 1e-4 * np.abs(w[fin]) + 1e-30)
    m, l, o, n = oracle.row_stats(post)
    st = buf.stats[0].cpu().numpy().reshape(-1, cfg.d + 4)
    assert np.array_equal(st[:, 2].astype(np.int64), n)
    assert np.all(np.abs(st[:, 0] - m) <= 1e-5 * np.abs(m) + 1e-6)
    assert np.all(np.abs(st[:, 1] - l) <= 1e-5 * l)
    assert np.all(np.linalg.norm(st[:, 4:] - o, axis=1) <= 1e-5 * np.linalg.norm(o, axis=1))


def test_infinite_value_row_stays_in_its_head():
    """An infinite value makes its KV head's effects non-finite or zero and
    leaves the other head's as they are without it."""
    cfg, tr = _case(dict(W=33, G=24))
    dev = DeviceTrajectory.upload(tr)
    buf = StepBuffers(cfg, [dev])
    head = [torch.zeros(cfg.M, cfg.Hq, dev.P_post, device="cuda")]
    out = []
    for _ in range(2):
        ck.commitkv_page_effects(buf.shape, [dev.post()], [buf.R_post[0]], head_R_out=head, workspace=buf.ws)
        assert buf.status() == ck.COMMITKV_OK
        out.append(head[0].cpu().numpy().copy())
        dev.post().v[0, 0, 70] = float("inf")
    g = cfg.Hq // cfg.H
    assert np.array_equal(out[0][:, g:], out[1][:, g:])
    assert np.isfinite(out[0]).any()


@pytest.mark.parametrize("off", ["pointer", "head stride"])
@pytest.mark.parametrize("d", [64, 128])
def test_a_pageless_cache_that_the_tensor_cores_cannot_read(d, off, monkeypatch):
    """The flash pass reads a cache without pages too (its row statistics): one
    element off a 16-byte boundary, or one head for all KV heads, sends its
    batch to the CUDA cores, as a cache with pages does."""
    M, H, S, W = 2, 2, 300, 8
    gen = torch.Generator("cuda").manual_seed(d)
    i32 = dict(dtype=torch.int32, device="cuda")
    pos = torch.arange(S, **i32)

    def cache(odd, pages):
        def values():
            flat = torch.randn(M * H * S * d + 1, generator=gen, device="cuda").bfloat16()
            if odd and off == "head stride":
                return flat[:M * S * d].view(M, 1, S, d).expand(M, H, S, d)
            return flat[int(odd):][:M * H * S * d].view(M, H, S, d)
        Q = torch.randn(M, 4, W, d, generator=gen, device="cuda").bfloat16()
        ps = torch.arange(0, 280 if pages else 0, 20, **i32)
        return ck.TrajTensors(values(), values(), pos, Q, pos[-W:].contiguous(), ps, torch.full_like(ps, 16))

    trajs = [cache(False, True), cache(True, False)]
    shape = ck.make_shape(M, H, 4, d, torch.bfloat16)
    ws = ck.alloc_workspace(shape, trajs)
    out = []
    for path in ("tc", "simt"):
        monkeypatch.setenv("COMMITKV_SCORING", path)
        R = [torch.zeros(t.page_start.numel(), device="cuda") for t in trajs]
        stats = torch.zeros(M, 4, W, d + 4, device="cuda")
        ck.commitkv_page_effects(shape, trajs, R, workspace=ws)
        ck.commitkv_page_effects(shape, trajs[1:], R[1:], stats_out=[stats], workspace=ws)
        assert ck.commitkv_workspace_status(ws) == ck.COMMITKV_OK
        out.append((R[0], stats))
    assert out[0][0].max() > 0 and torch.equal(out[0][0], out[1][0])
    assert out[0][1][..., 2].min() > 0 and torch.equal(out[0][1], out[1][1])
