"""The checkpoint's selection shares a trajectory's tokens between eight
blocks: indices equal to the oracle's at sizes around the shares and the
block's strides, with ties, retired and pending pages across the shares."""
import numpy as np
import pytest
import torch

from oracle import core
from paper_2608_07855_gb300 import commitkv as ck

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 7, 8, 9, 130, 1024, 8191, 8192, 8200, 20011])
@pytest.mark.parametrize("scores", ["uniform", "ties", "equal", "signs"])
def test_selection_over_eight_shares(S, scores):
    rng = np.random.default_rng(S)
    fill = {"uniform": rng.random(S), "ties": rng.integers(0, 5, S) / 4, "equal": np.full(S, 0.5),
            "signs": rng.standard_normal(S) * (rng.random(S) < 0.9)}[scores].astype(np.float32)
    ps = np.arange(0, S, 37, dtype=np.int32)
    pl = np.minimum(rng.integers(0, 38, len(ps)), S - ps).astype(np.int32)
    retired = (rng.random(len(ps)) < 0.2).astype(np.uint8)
    prio = rng.random(len(ps)).astype(np.float32)
    pending = np.flatnonzero(rng.random(len(ps)) < 0.5).astype(np.int32)
    i32 = dict(dtype=torch.int32, device="cuda")
    kv = torch.zeros(1, 1, S, 64, device="cuda")
    tr = ck.TrajTensors(kv, kv, torch.arange(S, **i32), None, None, torch.tensor(ps, **i32), torch.tensor(pl, **i32))
    shape = ck.make_shape(1, 1, 1, 64, torch.float32)
    ws = ck.alloc_workspace(shape, [tr, tr])
    for B in sorted({0, 1, S // 3, S - 1, S, S + 5}):
        B_N = B // 8
        idx = [torch.full((max(B, 1),), -1, **i32) for _ in range(2)]
        n = torch.zeros(2, **i32)
        dev = [torch.from_numpy(x).cuda() for x in (retired, pending, prio, fill)]
        ck.commitkv_compact(shape, [tr, tr], [dev[0]] * 2, [dev[1]] * 2, [dev[2]] * 2, [dev[3]] * 2, B, B_N, 16, idx, n,
                            workspace=ws)
        assert ck.commitkv_workspace_status(ws) == ck.COMMITKV_OK
        want = core.select_indices(S, ps, pl, retired, pending, prio[pending], fill, B, B_N, 16)
        for t in range(2):
            assert np.array_equal(idx[t].cpu().numpy()[:int(n[t])], want)
