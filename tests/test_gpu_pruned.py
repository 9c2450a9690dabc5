"""The pruned page pass scores only the (unit, page) pairs whose bound can
raise R, with the arithmetic of the full page pass: R is the same number,
bit for bit.  The full pass runs when maxima per head are asked for."""
import numpy as np
import pytest
import torch

from paper_2608_07855_gb300 import commitkv as ck

pytestmark = pytest.mark.gpu


def _pages(S, rng, sizes, gap):
    ps, pl, t = [], [], int(rng.integers(0, 40))
    while True:
        n = int(rng.choice(sizes))
        if t + n > S:
            break
        ps.append(t)
        pl.append(n)
        t += n + (int(rng.integers(0, gap + 1)) if rng.random() < 0.3 else 0)
    return ps, pl


def _traj(M, H, Hq, d, S, W, sizes, kind, seed, gap=60):
    gen = torch.Generator("cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)

    def normal(*s):
        return torch.randn(*s, generator=gen, device="cuda")

    K, V, Q = normal(M, H, S, d), normal(M, H, S, d), normal(M, Hq, W, d)
    if kind == "sharp":  # a few tokens hold nearly all of some rows' attention
        K[:, :, :: max(S // 7, 1)] *= 6.0
    elif kind == "uniform":  # every share alike: no bound is far from the effect
        K.zero_()
    elif kind == "zero_v":
        V.zero_()
    elif kind == "small":  # squares of the values underflow
        V *= 1e-21
    elif kind == "big_v":  # norms above the range of 16-bit floats
        V *= 3e5
    elif kind == "inf_v":
        V[0, 0, S // 2] = float("inf")
    elif kind == "nan_k":
        K[M - 1, 0, S // 3, 0] = float("nan")
    pos = torch.cumsum(torch.randint(1, 3, (S,), generator=gen, device="cuda"), 0).int()
    last = int(pos[-1])
    qpos = torch.arange(last - W + 1, last + 1, dtype=torch.int32, device="cuda")
    if kind == "blind":  # the first window position sees nothing
        qpos[0] = -5
    ps, pl = _pages(S, rng, sizes, gap)
    i32 = dict(dtype=torch.int32, device="cuda")
    return ck.TrajTensors(K.bfloat16(), V.bfloat16(), pos, Q.bfloat16(), qpos, torch.tensor(ps, **i32),
                          torch.tensor(pl, **i32))


CASES = [
    # M, H, Hq, W, S, page sizes, kind; each over the amount of work from which the page pass is pruned
    (64, 8, 32, 16, 2100, [32], "normal"),
    (64, 8, 32, 32, 2113, [16], "sharp"),
    (64, 8, 64, 20, 1500, [8, 9, 127, 128, 129, 300], "normal"),  # 160 rows: a ragged second row tile
    (64, 8, 16, 8, 2200, [0, 32, 33], "sharp"),
    (128, 8, 32, 16, 1100, [32], "uniform"),
    (256, 16, 32, 32, 300, [16], "zero_v"),
    (256, 8, 16, 8, 513, [16, 40], "small"),
    (256, 8, 16, 8, 512, [64], "big_v"),
    (128, 8, 16, 8, 1100, [32], "inf_v"),
    (128, 8, 16, 8, 1100, [32], "nan_k"),
    (256, 8, 16, 4, 600, [32], "blind"),
    (64, 8, 16, 4, 3000, [2800], "sharp"),  # one page of many tiles holding almost everything
    (64, 8, 16, 8, 2100, [2, 3], "normal"),
    (64, 8, 16, 8, 2100, [1, 2], "normal"),  # pages too short to prune: the full pass both times
    (128, 16, 32, 32, 1500, [16], "uniform"),  # units that keep everything, enough of them for items of two buckets
    (128, 16, 32, 32, 2300, [16], "uniform"),  # the same with a third bucket alone
]


def _both(trajs, M, Hq, mask=None, prunes=True, most=1.0):
    """R with the pruned page pass and with the full one, as bits.  `prunes`:
    whether the first call prunes; then at most the share `most` of the (row
    tile, page) pairs is scored."""
    shape = ck.make_shape(M, trajs[0].k.shape[1], Hq, trajs[0].k.shape[3], torch.bfloat16)
    ws = ck.alloc_workspace(shape, trajs)
    out = []
    for head in (False, True):
        R = [torch.full((t.page_start.numel(),), -1.0, device="cuda") for t in trajs]
        hR = [torch.zeros(M, Hq, t.page_start.numel(), device="cuda") for t in trajs] if head else None
        ck.commitkv_page_effects(shape, trajs, R, head_R_out=hR, layer_mask=mask, workspace=ws)
        scored = sum(ck.commitkv_test_pruned_pages(ws))
        tiles = [-(-Hq // shape.kv_heads * t.q.shape[2] // 128) * t.page_start.numel() for t in trajs]
        assert (scored > 0) == (prunes and not head)
        assert scored <= most * M * shape.kv_heads * sum(tiles)
        assert ck.commitkv_workspace_status(ws) == ck.COMMITKV_OK
        out.append([r.cpu().numpy().view(np.uint32) for r in R])
    return out


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[6]}-{c[4]}-{c[5][0]}")
def test_pruned_effects_equal_the_full_pass(case, d):
    M, H, Hq, W, S, sizes, kind = case
    short, whole = sizes == [1, 2], (sizes, kind) == ([16], "uniform")
    t = _traj(M, H, Hq, d, S, W, sizes, kind, d + 1, 0 if short or whole else 60)
    assert (2 * t.page_start.numel() > S) == short
    if whole:  # eight items of 128 slots a SM, from units that drop nothing
        slots = int(((t.page_len + 15) // 16).sum()) * M * H * (-(-Hq // H * W // 128))
        assert slots >= 8 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    # a fifth to three fifths is scored of the sharp caches with many pages, a hundredth of short pages
    most = 0.75 if kind == "sharp" and len(t.page_start) > 1 else 0.05 if sizes == [2, 3] else 1.0
    pruned, full = _both([t], M, Hq, prunes=not short, most=most)
    assert np.array_equal(pruned[0], full[0])


def test_pruned_effects_of_a_ragged_batch_with_a_layer_mask():
    sizes = [300, 2000, 129, 777, 1300]
    trajs = [_traj(256, 2, 8, 128, S, W, [16, 32], "sharp", i) for i, (S, W) in enumerate(zip(sizes, [8, 32, 4, 40, 16]))]
    none = torch.zeros(0, dtype=torch.int32, device="cuda")
    trajs.append(ck.TrajTensors(trajs[0].k, trajs[0].v, trajs[0].pos, trajs[0].q, trajs[0].q_pos, none, none))
    for mask in (None, [0, 1] * 128):
        pruned, full = _both(trajs, 256, 8, mask)
        for a, b in zip(pruned, full):
            assert np.array_equal(a, b)


def test_pruned_effects_of_two_launches():
    """18 caches take two launches, which use one region of tables in turn."""
    trajs = [_traj(128, 8, 16, 128, 140 + 7 * i if i < 16 else 700 + i, 8, [16], "sharp", i, 4) for i in range(18)]
    pruned, full = _both(trajs, 128, 16)
    for a, b in zip(pruned, full):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("M,H,Hq,d,dtype,S,W,P,size", [(64, 8, 32, 128, "bfloat16", 2200, 8, 130, 112596992),
                                                       (16, 2, 8, 64, "bfloat16", 2200, 8, 130, 3064320),
                                                       (1, 2, 4, 64, "float32", 2300, 16, 140, 192000)],
                         ids=["pruned", "64channels", "small-f32"])
def test_a_workspace_without_room_for_the_faster_path(M, H, Hq, d, dtype, S, W, P, size):
    """`size` is what commitkv_workspace_size gave before there were bounds,
    64-channel tensor-core kernels and short chunks of small calls: such a
    buffer still serves, and a quarter of it is refused as before."""
    t = _traj(M, H, Hq, d, S, W, [16], "normal", 7)
    dt = getattr(torch, dtype)
    t = ck.TrajTensors(t.k.to(dt), t.v.to(dt), t.pos, t.q.to(dt), t.q_pos, t.pos[:0].new_tensor(range(0, 16 * P, 16)),
                       t.pos.new_full((P,), 16))
    shape = ck.make_shape(M, H, Hq, d, dt)
    out = []
    for n in (ck.commitkv_workspace_size(shape, [t]), size):
        ws = torch.empty(n + 512, dtype=torch.uint8, device="cuda")
        ws[n:] = 0x5A  # past the end
        ck.commitkv_workspace_init(ws[:n])
        R = torch.zeros(P, device="cuda")
        ck.commitkv_page_effects(shape, [t], [R], workspace=ws[:n])
        pages = ck.commitkv_test_pruned_pages(ws[:n])
        assert ck.commitkv_workspace_status(ws[:n]) == ck.COMMITKV_OK
        assert bool((ws[n:] == 0x5A).all())
        out.append((n, pages, R))
    assert out[0][0] > size
    assert (sum(out[0][1]) > 0) == (d == 128) and sum(out[1][1]) == 0
    a, b = out[0][2], out[1][2]
    if d == 128:  # the same values
        assert torch.equal(a, b)
    else:  # each within 1e-4 of the exact effects (the bound of both paths' tests)
        assert torch.isfinite(a).all() and ((a - b).abs() <= 2e-4 * a).all()
    with pytest.raises(RuntimeError):
        ck.commitkv_page_effects(shape, [t], [R], workspace=torch.empty(size // 4 // 256 * 256, dtype=torch.uint8, device="cuda"))


def test_a_nan_effect_ranks_above_an_infinite_one():
    """The first page is all that the first window position sees (effect
    infinite in every unit), and one head's values make its other rows'
    effects NaN: a unit with an infinite bound is scored although R is
    infinite already."""
    t = _traj(128, 8, 16, 128, 1100, 64, [32], "normal", 5)
    n = int(t.page_start[0] + t.page_len[0])
    t.page_start[0], t.page_len[0] = 0, n
    t.q_pos[0] = t.pos[n - 1]
    t.v[0, 0, 3, 5] = float("inf")
    pruned, full = _both([t], 128, 16)
    assert np.isnan(full[0].view(np.float32)[0]) and np.array_equal(pruned[0], full[0])


@pytest.mark.parametrize("Hq,W", [(32, 8), (64, 20)], ids=["32rows", "160rows"])
@pytest.mark.parametrize("d", [128, 64])
def test_what_the_workspace_held_does_not_change_what_is_scored(d, Hq, W):
    """A row tile that the probe rows fill in part: of the rows past their end
    nothing is written, and the bounds may not read them (0xff and 0x7e bytes
    are NaN as 16-bit floats, 0x7c an infinity or a NaN)."""
    M, H, S = 64, 8, 2200
    t = _traj(M, H, Hq, d, S, W, [16], "sharp", 11)
    shape = ck.make_shape(M, H, Hq, d, torch.bfloat16)
    ws = ck.alloc_workspace(shape, [t])
    P, seen = t.page_start.numel(), []
    for byte in (0, 0xFF, 0x7E, 0x7C):
        ws[256:] = byte
        R = torch.zeros(P, device="cuda")
        ck.commitkv_page_effects(shape, [t], [R], workspace=ws)
        pages = ck.commitkv_test_pruned_pages(ws)
        assert ck.commitkv_workspace_status(ws) == ck.COMMITKV_OK
        seen.append((pages, R.cpu().numpy().tobytes()))
    assert 0 < sum(seen[0][0]) < M * H * ((Hq // H * W + 127) // 128) * P
    assert all(s == seen[0] for s in seen)


def test_overlapping_pages_are_reported_and_stay_in_bounds():
    """A zero-length page between two pages of the same span: each is
    compared with every earlier page, not with its neighbour alone."""
    t = _traj(128, 8, 16, 128, 1100, 8, [32], "normal", 3)
    i32 = dict(dtype=torch.int32, device="cuda")
    t.page_start = torch.tensor([0, 0, 0, 0, 0, 1080], **i32)
    t.page_len = torch.tensor([1000, 0, 1000, 0, 1000, 12], **i32)
    shape = ck.make_shape(128, 8, 16, 128, torch.bfloat16)
    ws = ck.alloc_workspace(shape, [t])
    for head in (None, [torch.zeros(128, 16, 6, device="cuda")]):
        R = torch.zeros(6, device="cuda")
        ck.commitkv_page_effects(shape, [t], [R], head_R_out=head, workspace=ws)
        assert ck.commitkv_workspace_status(ws) == ck.COMMITKV_ERR_DEVICE_INPUT
