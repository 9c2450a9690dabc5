"""Kernels launched per step, as the library counts them and the benchmark
reports them: classify two (states, order), joint test two (clears, scan),
compaction two (selection, gather), and the scoring call's own."""
import dataclasses

import pytest
import torch

from paper_2608_07855_gb300 import commitkv as ck
from paper_2608_07855_gb300 import synth
from paper_2608_07855_gb300.workload import DeviceTrajectory, StepBuffers

pytestmark = pytest.mark.gpu

REST = 2 + 2 + 2
TC = 4            # prep, flash pass, combine, page pass
PRUNED = 3 + 6    # bounds, seeds, and two lists with a page pass each take the page pass's place
SIMT = 4          # visible counts, flash pass, combine, page pass
# 17 caches make two launch sequences on the tensor cores; with 64 channels the
# pre-commit caches take the tensor cores and the post-commit ones the CUDA cores
CASES = [("f32", dict(dtype="f32", d=64, outlier_channels=0), 1, SIMT), ("bf16", dict(), 1, TC), ("batch", dict(), 9, 2 * TC),
         ("64channels", dict(d=64), 1, TC + SIMT), ("pruned", dict(M=128, H=8, Hq=8, L_pre=900, L_obs=100), 1, PRUNED)]


@pytest.mark.parametrize("name,kw,n,score", CASES, ids=[c[0] for c in CASES])
def test_launches_of_a_step(name, kw, n, score):
    cfg = dataclasses.replace(synth.small_config(name, **kw), n_traj=n)
    buf = StepBuffers(cfg, [DeviceTrajectory.upload(synth.make_trajectory(cfg, 0, traj=t)) for t in range(n)])
    for _ in range(2):
        before = ck.commitkv_test_launches()
        buf.step()
        assert ck.commitkv_test_launches() - before == score + REST
    torch.cuda.synchronize()
    assert buf.status() == ck.COMMITKV_OK
