"""Performance cases of the library: what each measures, and how its inputs and exact results are made.

A case is one pass through the Python binding's public entry points (`paper_2608_07855_gb300.commitkv`, `workload`,
`lifecycle`) on a seeded synthetic agent trajectory: events of 32 to 256 tokens in turn (reasoning, tool call,
observation), the tool calls and observations cut into G-token pages, then the returned observation and the W decoded
tokens of the post-commit window.  K, V, Q are N(0, 1) with four outlier key channels per KV head and one shared query
direction per window; a fifth of the pages have keys that one pre-commit probe query attends to and the post-commit
window turns away from (the high-to-low pages); each holds about half of that query's attention.

Fields: op, dtype, d (head width), M layers, H KV heads, Hq query heads, W probe positions, G page tokens, ctx and obs
(tokens before the commit, tokens of the observation; the largest ones when n > 1), n trajectories, B budget, sel (0:
all layers take part, else that many of them), layout (the seed of event lengths, so that a case's work is fixed)."""
import math
import random

import torch

from paper_2608_07855_gb300 import commitkv as ck
from paper_2608_07855_gb300.lifecycle import Session
from paper_2608_07855_gb300.synth import Config
from paper_2608_07855_gb300.workload import DeviceTrajectory, StepBuffers

BETA, GAMMA, SIGMA, NU = (8.0, 12.0), 8.0, 0.25, 6.0
TAU = 0.03  # bound of the joint test
NEW = 128  # decoded tokens between two checkpoints of a session


def _case(name, op, ctx, obs, dtype="bf16", d=128, M=36, H=8, Hq=32, W=32, G=32, n=1, B=4096, sel=0, layout=1):
    return dict(name=name, op=op, dtype=dtype, d=d, M=M, H=H, Hq=Hq, W=W, G=G, ctx=ctx, obs=obs, n=n, B=B, sel=sel,
                layout=layout)


def listed():
    return [
        # the smallest: a whole step on the one-layer fp32 reference workload, where launches and host time count
        _case("step_tiny_f32", "step", 2048, 256, "f32", 64, 1, 2, 4, 16, 16, B=1024),
        # the benchmark's own workload: a whole step (score, classify, joint test, compact) at 32K + 4K
        _case("step_8b_32k", "step", 32768, 4096, B=8192),
        # both scoring passes of one commit at the ordinary context length
        _case("effects_8b_16k", "effects", 16384, 2048),
        # concurrent agents with contexts of very different lengths, scored in one call
        _case("effects_ragged_8", "effects", 32768, 4096, n=8, layout=4),
        # the largest: 64 layers, 64 query heads, 64 probe positions, 128K context; bound by arithmetic
        _case("effects_32b_128k", "effects", 131072, 8192, M=64, Hq=64, W=64, G=64),
        # an early turn with the paper's own window and page size (W = 8, G = 16): little work in many small pages
        _case("effects_early_turn", "effects", 1931, 517, W=8, G=16, layout=2),
        # a model with 64-wide heads in bf16
        _case("effects_d64", "effects", 8192, 1024, d=64, M=16, layout=3),
        # an engine that already has the window's output and log-sum-exp; ragged length
        _case("from_stats_8b_24k", "from_stats", 23457, 2983, layout=5),
        # fill scores of a long cache
        _case("token_scores_8b_32k", "tokens", 32768, 4096, layout=6),
        # the greedy scan over the candidates of a commit
        _case("joint_8b_20k", "joint", 20011, 2500, layout=7),
        # a checkpoint into new buffers
        _case("compact_8b_32k", "compact", 32768, 4096, B=8192, layout=8),
        # the most frequent call of a session: 128 decoded tokens appended, fill scores, in-place checkpoint
        _case("session_checkpoint_4k", "session", 4096 + NEW, 0, B=4096, layout=9),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "effects", "effects", "effects", "from_stats", "tokens", "joint", "compact", "session"])
    kind = rng.choice(["8b", "8b", "8b", "32b", "d64", "f32"])
    c = dict(op=op, dtype="bf16", d=128, M=36, H=8, Hq=32, W=rng.choice([8, 16, 32, 32, 31]), G=rng.choice([16, 32, 32, 64]),
             n=1, sel=rng.choice([0, 0, 0, 1, 5]), layout=rng.randrange(1 << 20))
    ctx = _log(rng, 1200, 32768)
    if kind == "32b":
        c.update(M=64, Hq=64, W=64, G=64)
    elif kind == "d64":
        c.update(d=64, M=rng.choice([12, 16, 24]), H=rng.choice([2, 4, 8]))
        ctx = _log(rng, 1200, 12000)
    elif kind == "f32":
        H = rng.choice([2, 4])
        c.update(dtype="f32", d=rng.choice([64, 128]), M=rng.choice([1, 2, 4]), H=H, Hq=H * rng.choice([2, 4]), G=16)
        ctx = _log(rng, 1200, 6000)
    if op == "effects" and kind == "8b" and rng.random() < 0.4:
        c["n"], ctx = rng.randint(2, 8), _log(rng, 4096, 32768)
    c["ctx"], c["obs"] = ctx, max(64, int(ctx * rng.uniform(0.05, 0.3)))
    c["B"] = max(256, int(ctx * rng.uniform(0.15, 0.5)))
    if op in ("step", "compact", "session"):
        c["sel"] = 0
    if op == "session":
        c["ctx"], c["obs"], c["B"] = ctx // 4 + 768 + NEW, 0, ctx // 4 + 768
    return c


# ------------------------------------------------------------------------------------------------ layout
def _layouts(c):
    """Per trajectory: (L_pre, L_obs, page starts, page lengths, pages resident before the commit)."""
    rng = random.Random(c["layout"])
    out = []
    for _ in range(c["n"]):
        L = c["ctx"] if c["n"] == 1 else rng.randint(c["ctx"] // 8, c["ctx"])
        obs = c["obs"] if c["n"] == 1 else rng.randint(c["obs"] // 16, c["obs"])
        a = rng.randint(32, 256)  # the current tool call ends the pre-commit cache
        events, t, j = [], 0, 0
        while t < L - a:
            m = min(rng.randint(32, 256), L - a - t)
            events.append((j % 3 > 0, t, m))
            t, j = t + m, j + 1
        events.append((True, L - a, a))
        if obs:
            events.append((True, L, obs))
        ps, pl = [], []
        for paged, b, m in events:
            for s in range(b, b + m, c["G"]) if paged else ():
                ps.append(s)
                pl.append(min(c["G"], b + m - s))
        out.append((L, obs, ps, pl, sum(1 for s in ps if s < L)))
    return out


def _planted(c, lay):
    """The high-to-low pages: a fifth of those resident before the commit, the last events left out."""
    ps, P_pre = lay[2], lay[4]
    pool = [E for E in range(P_pre) if ps[E] < lay[0] - 320]
    rng = random.Random(c["layout"] * 7 + 1 + lay[0])
    return sorted(rng.sample(pool, min(len(pool), max(1, P_pre // 5))))


def _betas(planted, seed, t):
    """How far the post-commit window turns away from each planted page."""
    rng = random.Random(seed * 31 + t)
    return [rng.uniform(*BETA) for _ in planted]


def _layers(c):
    """The mask of the layers that take part, or None."""
    if not c["sel"] or c["sel"] >= c["M"]:
        return None
    pick = {i * c["M"] // c["sel"] for i in range(c["sel"])}
    return [l in pick for l in range(c["M"])]


def _n_layers(c):
    m = _layers(c)
    return sum(m) if m else c["M"]


# ------------------------------------------------------------------------------------------------ inputs
def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _values(c, lay, seed, t):
    """K, V [M][H][S][d], Q- and Q+ [M][Hq][W][d] of one trajectory, on the GPU."""
    M, H, Hq, d, W = c["M"], c["H"], c["Hq"], c["d"], c["W"]
    g, dt = Hq // H, torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    gen = torch.Generator("cuda").manual_seed(seed * 1009 + t)

    def normal(*shape, dtype=torch.float32):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=dtype)

    L, obs, ps, pl, P_pre = lay
    S = L + obs + W
    K, V = normal(M, H, S, d, dtype=dt), normal(M, H, S, d, dtype=dt)
    scale = torch.ones(M, H, 1, d, device="cuda", dtype=dt)
    loud = torch.rand(M, H, 1, d, generator=gen, device="cuda").topk(4, dim=-1).indices
    K *= scale.scatter_(3, loud, 8.0 if c["dtype"] == "bf16" else 1.0)
    cm = _unit(normal(M, H, d))
    cp = normal(M, H, d)
    cp = _unit(cp - (cp * cm).sum(-1, keepdim=True) * cm)
    Qm = normal(M, H, g * W, d) + GAMMA * cm[:, :, None]
    Qp = normal(M, H, g * W, d) + GAMMA * cp[:, :, None]
    planted = _planted(c, lay)
    tok = torch.tensor([i for E in planted for i in range(ps[E], ps[E] + pl[E])], dtype=torch.long, device="cuda")
    page = torch.tensor([j for j, E in enumerate(planted) for _ in range(pl[E])], dtype=torch.long, device="cuda")
    beta = torch.tensor(_betas(planted, seed, t), device="cuda")
    row = torch.randint(0, g * W, (M, H, len(planted)), generator=gen, device="cuda")
    u = Qm.gather(2, row[..., None].expand(-1, -1, -1, d))
    for x in (cp, cm):
        u = u - (u * x[:, :, None]).sum(-1, keepdim=True) * x[:, :, None]
    # exp(alpha) on each of the page's tokens is about the sum over the rest of the cache
    u = math.log(4 * L / c["G"]) * _unit(u) - beta[None, None, :, None] * cp[:, :, None]
    for l in range(M):  # layer by layer: the rows of many planted tokens are large
        K[l][:, tok] = (u[l][:, page] + SIGMA * normal(H, len(tok), d)).to(dt)
        V[l][:, tok] += (NU * _unit(normal(H, 1, d))).to(dt)
    return K, V, Qm.view(M, Hq, W, d).to(dt), Qp.view(M, Hq, W, d).to(dt)


class _Layout:
    """What StepBuffers reads of a trajectory's host description."""

    def __init__(self, lay):
        self.L_pre, self.P_pre, self.P_post = lay[0], lay[4], len(lay[2])


def _trajectories(c, seed):
    i32 = dict(dtype=torch.int32, device="cuda")
    out = []
    for t, lay in enumerate(_layouts(c)):
        L, obs, ps, pl, P_pre = lay
        K, V, Qm, Qp = _values(c, lay, seed, t)
        S = K.shape[2]
        gen = torch.Generator("cuda").manual_seed(seed * 1013 + t)
        eligible = torch.zeros(len(ps), dtype=torch.uint8, device="cuda")
        eligible[:P_pre] = 1
        out.append(DeviceTrajectory(
            _Layout(lay), K, V, torch.arange(S, **i32), Qm, Qp, torch.arange(L - c["W"], L, **i32),
            torch.arange(L + obs, S, **i32), torch.tensor(ps, **i32), torch.tensor(pl, **i32), eligible,
            torch.arange(P_pre, len(ps), **i32), torch.rand(S, generator=gen, device="cuda")))
    return out


def _config(c):
    return Config("case", M=c["M"], H=c["H"], Hq=c["Hq"], d=c["d"], dtype=c["dtype"], L_pre=c["ctx"], L_obs=c["obs"],
                  W=c["W"], G=c["G"], B=c["B"], tau_joint=TAU, pending_cap=16)


def _row_stats(q, k, v, pos, qpos, dtype):
    """m, l, n, o of every probe row: q [H][rows][d], k, v [H][S][d], qpos [rows]; [H][rows][d + 4]."""
    q, k, v = q.to(dtype), k.to(dtype), v.to(dtype)
    s = (q @ k.mT) / math.sqrt(q.shape[-1])
    seen = pos[None, :] <= qpos[:, None]
    s.masked_fill_(~seen, -math.inf)
    m = s.amax(-1, keepdim=True)
    e = s.sub_(m).exp_()
    l = e.sum(-1, keepdim=True)
    n = seen.sum(-1).to(dtype)[None, :, None].expand(q.shape[0], -1, 1)
    return torch.cat([m, l, n, torch.zeros_like(n), (e @ v) / l], -1), e


def _stats(c, t):
    """Row statistics [M][Hq][W][d + 4] of the post-commit window, by plain torch in 32 bits."""
    M, H, Hq, d, W = c["M"], c["H"], c["Hq"], c["d"], c["W"]
    qpos = t.qpos_post.repeat(Hq // H)
    rows = [_row_stats(t.Q_post[l].view(H, -1, d), t.K[l], t.V[l], t.pos, qpos, torch.float32)[0] for l in range(M)]
    return torch.stack(rows).view(M, Hq, W, d + 4).contiguous()


def prepare(case, seed):
    c = case
    if c["op"] == "session":
        return _prepare_session(c, seed)
    trajs = _trajectories(c, seed)
    st = dict(case=c, trajs=trajs, mask=_layers(c))
    buf = st["buf"] = StepBuffers(_config(c), trajs) if c["op"] in ("step", "compact") else None
    if buf is not None:
        if c["op"] == "compact":  # the pages that an earlier joint test accepted, the effects of an earlier pass
            gen = torch.Generator("cuda").manual_seed(seed)
            for t, lay in enumerate(_layouts(c)):
                buf.accepted[t][torch.tensor(_planted(c, lay), device="cuda")[::2]] = 1
                buf.R_post[t].copy_(torch.rand(len(lay[2]), generator=gen, device="cuda"))
        return st
    st["shape"] = ck.make_shape(c["M"], c["H"], c["Hq"], c["d"], trajs[0].K.dtype)
    st["pre"], st["post"] = [t.pre() for t in trajs], [t.post() for t in trajs]
    st["ws"] = ck.alloc_workspace(st["shape"], st["pre"] + st["post"])
    f32 = dict(dtype=torch.float32, device="cuda")
    st["R_pre"] = [torch.zeros(t.P_pre, **f32) for t in trajs]
    st["R_post"] = [torch.zeros(t.P_post, **f32) for t in trajs]
    if c["op"] == "effects":
        st["stats"] = [torch.zeros(c["M"], c["Hq"], c["W"], c["d"] + 4, **f32) for t in trajs]
        return st
    st["stats"] = [_stats(c, t) for t in trajs]
    if c["op"] == "tokens":
        st["scores"] = [torch.zeros(t.pos.numel(), **f32) for t in trajs]
    if c["op"] == "joint":
        st["cand"] = []
        for t, lay in enumerate(_layouts(c)):  # by growing effect on the window, as classify orders them
            cand = torch.zeros(len(lay[2]), dtype=torch.int32, device="cuda")
            planted = _planted(c, lay)
            pages = [E for _, E in sorted(zip(_betas(planted, seed, t), planted), reverse=True)]
            cand[:len(pages)] = torch.tensor(pages, dtype=torch.int32)
            st["cand"].append(cand)
        st["n_cand"] = torch.tensor([len(_planted(c, lay)) for lay in _layouts(c)], dtype=torch.int32, device="cuda")
        st["accepted"] = [torch.zeros(t.P_post, dtype=torch.uint8, device="cuda") for t in trajs]
        st["step_R"] = [torch.zeros(t.P_post, **f32) for t in trajs]
    return st


def _prepare_session(c, seed):
    """A session after a commit and the checkpoint that filled its cache up to the budget, and the next NEW tokens."""
    B, W, lay = c["B"], c["W"], _layouts(c)[0]
    n = B + NEW
    K, V, Qm, Qp = _values(c, lay, seed, 0)
    s = Session(ck.make_shape(c["M"], c["H"], c["Hq"], c["d"], K.dtype), c["G"], B, 0.125, n)
    pos = torch.arange(n, dtype=torch.int32, device="cuda")
    s.append(K[:, :, :n], V[:, :, :n], pos, [("call", b, m) for b, m in zip(lay[2], lay[3])])
    s.pre_commit(Qm, pos[n - W:])
    s.post_commit(Qp, pos[n - W:])
    s.decode_checkpoint(Qp, pos[n - W:])
    gen = torch.Generator("cuda").manual_seed(seed * 1019)
    new = [torch.randn(c["M"], c["H"], NEW, c["d"], generator=gen, device="cuda", dtype=K.dtype) for _ in range(2)]
    return dict(case=c, session=s, Q=Qp, new=new, at=n)


def _parts(stats):
    """The row statistics' columns by kind: the visible counts are far larger than the rest."""
    return dict(m=[s[..., 0] for s in stats], l=[s[..., 1] for s in stats], n=[s[..., 2] for s in stats],
                o=[s[..., 4:] for s in stats])


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "step":
        b = state["buf"]
        b.step()
        return dict(R_pre=b.R_pre, R_post=b.R_post, **_parts(b.stats), state=b.state, cand=b.cand, n_cand=b.n_cand,
                    accepted=b.accepted, step_R=b.step_R, idx=b.idx, n_idx=b.n_idx, k=b.k_out, v=b.v_out, pos=b.pos_out)
    if op == "compact":
        b = state["buf"]
        b.compact()
        return dict(idx=b.idx, n_idx=b.n_idx, k=b.k_out, v=b.v_out, pos=b.pos_out)
    if op == "session":
        s, at, W = state["session"], state["at"], c["W"]
        pos = torch.arange(at, at + NEW, dtype=torch.int32, device="cuda")
        s.append(state["new"][0], state["new"][1], pos, [("call", at + 20, 70)], decoded=NEW)
        state["at"] = at + NEW
        scores = s.fill_scores(state["Q"], pos[NEW - W:])
        idx = s.checkpoint(scores)
        n = idx.numel()
        return dict(scores=scores, idx=idx, k=s.K[:, :, :n], v=s.V[:, :, :n], pos=s.pos[:n],
                    pages=[x for p in s.pages[:8] for x in p])
    shape, ws, mask = state["shape"], state["ws"], state["mask"]
    if op == "effects":
        ck.commitkv_page_effects(shape, state["pre"] + state["post"], state["R_pre"] + state["R_post"],
                                 stats_out=[None] * c["n"] + state["stats"], layer_mask=mask, workspace=ws)
        return dict(R_pre=state["R_pre"], R_post=state["R_post"], **_parts(state["stats"]))
    if op == "from_stats":
        ck.commitkv_page_effects_from_stats(shape, state["post"], state["stats"], state["R_post"], layer_mask=mask,
                                            workspace=ws)
        return dict(R_post=state["R_post"])
    if op == "tokens":
        ck.commitkv_token_scores(shape, state["post"], state["stats"], state["scores"], layer_mask=mask, workspace=ws)
        return dict(scores=state["scores"])
    ck.commitkv_joint_test(shape, state["post"], state["stats"], state["cand"], state["n_cand"], TAU, state["accepted"],
                           state["step_R"], layer_mask=mask, workspace=ws)
    return dict(accepted=state["accepted"], step_R=state["step_R"])


# ------------------------------------------------------------------------------------------------ work
def work(case):
    """Each token's K and V read once, each retained row read and written once, statistics read or written once."""
    c = case
    es, nl = (2 if c["dtype"] == "bf16" else 4), _n_layers(c)
    row = c["H"] * c["d"] * es  # one token of K (or V) in one layer
    dots = 2.0 * c["Hq"] * c["W"] * c["d"]  # one token against every probe row of one layer, one product
    q = c["Hq"] * c["W"] * c["d"] * es
    stats = c["Hq"] * c["W"] * (c["d"] + 4) * 4
    lays = _layouts(c)
    pre, post = sum(x[0] for x in lays), sum(x[0] + x[1] + c["W"] for x in lays)
    paged, op = sum(sum(x[3]) for x in lays), c["op"]
    move = 2.0 * c["B"] * 2 * row * c["M"] * c["n"]  # a retained row: K and V, read and written
    if op in ("effects", "step"):
        b = nl * ((pre + post) * 2 * row + c["n"] * (2 * q + stats)) + (move if op == "step" else 0)
        return dict(bytes=b, flops=nl * (pre + post) * 2 * dots)
    if op == "from_stats":
        return dict(bytes=nl * (paged * 2 * row + q + stats), flops=nl * paged * 2 * dots)
    if op == "tokens":
        return dict(bytes=nl * (post * row + q + stats) + post * 4, flops=nl * post * dots)
    if op == "joint":
        cand = sum(lay[3][E] for lay in lays for E in _planted(c, lay))
        return dict(bytes=nl * (cand * 2 * row + q + stats), flops=nl * cand * 2 * dots)
    if op == "compact":
        return dict(bytes=move + post * 4, flops=0)
    S = c["B"] + NEW  # a session: the cache read once for the scores, 128 tokens appended, the survivors moved
    return dict(bytes=c["M"] * (S * 2 * row + 2 * NEW * 2 * row) + move, flops=c["M"] * S * 2 * dots)


def tolerance(case):
    """Four times what the same arithmetic in another order gives; `differ`: retained tokens, states and candidates
    whose scores are equal to rounding."""
    if case["op"] == "compact":
        return "exact"
    if case["dtype"] == "f32":
        return dict(rel=1e-5, max=4e-4, differ=0.01)
    return dict(rel=1e-4, max=4e-3, differ=0.01)


# ------------------------------------------------------------------------------------------------ exact
def _effects64(c, lay, K, V, Q, pos, qpos, P, mask):
    """R [P] and the statistics [M][Hq][W][d + 4] in 64 bits: the definition's closed form, one KV head at a time."""
    f64 = torch.float64
    M, H, Hq, d, W = c["M"], c["H"], c["Hq"], c["d"], c["W"]
    ps = torch.tensor(lay[2][:P], device="cuda")
    pl = torch.tensor(lay[3][:P], device="cuda")
    col = torch.arange(c["G"], device="cuda")
    tok = (ps[:, None] + col).clamp(max=K.shape[2] - 1)
    live = (col[None, :] < pl[:, None]).to(f64)
    R = torch.zeros(P, dtype=f64, device="cuda")
    stats = torch.zeros(M, Hq, W, d + 4, dtype=f64, device="cuda")
    rows_pos = qpos.repeat(Hq // H)
    for l in range(M):
        if mask and not mask[l]:
            continue
        for h in range(H):
            q = Q[l].view(H, -1, d)[h:h + 1]
            st, e = _row_stats(q, K[l, h:h + 1], V[l, h:h + 1], pos, rows_pos, f64)
            st, e = st[0], e[0]
            stats[l].view(H, -1, d + 4)[h] = st
            o, lsum, norm = st[:, 4:], st[:, 1], st[:, 4:].norm(dim=-1)
            ep = (e[:, tok] * live).transpose(0, 1)  # [P][rows][G]
            S = ep.sum(-1)
            D = ep @ V[l, h].to(f64)[tok]
            D -= S[..., None] * o
            R = torch.maximum(R, (D.norm(dim=-1) / ((lsum - S) * norm)).amax(-1))
    return R, stats


def _joint64(c, lay, t, stats, cand, mask):
    """The scan's step values in 64 bits, from the same row statistics."""
    M, H, Hq, d = c["M"], c["H"], c["Hq"], c["d"]
    f64 = torch.float64
    layers = [l for l in range(M) if not mask or mask[l]]
    rows_pos = t.qpos_post.repeat(Hq // H)
    st = stats.view(M, H, -1, d + 4)[layers].to(f64)  # [layers][H][rows]
    q = t.Q_post.view(M, H, -1, d)[layers].to(f64)
    m, lsum, o = st[..., 0], st[..., 1], st[..., 4:]
    norm = o.norm(dim=-1)
    DA, SA, steps = torch.zeros_like(o), torch.zeros_like(lsum), []
    for E in cand:
        b, n = lay[2][E], lay[3][E]
        e = torch.einsum("lhrd,lhid->lhri", q, t.K[layers, :, b:b + n].to(f64)) / math.sqrt(d)
        e = (e - m[..., None]).exp() * (t.pos[b:b + n][None, :] <= rows_pos[:, None])
        D = DA + e @ t.V[layers, :, b:b + n].to(f64) - e.sum(-1)[..., None] * o
        S = SA + e.sum(-1)
        steps.append(float((D.norm(dim=-1) / ((lsum - S) * norm)).max()))
        if steps[-1] <= TAU:
            DA, SA = D, S
    return torch.tensor(steps + [0.0] * (len(lay[2]) - len(cand)), dtype=f64)


def exact(case, seed):
    c = case
    if c["op"] == "compact" or work(c)["flops"] > 1.2e13:  # copies; over 20 seconds in 64 bits
        return None
    if c["op"] == "session":
        st = prepare(c, seed)
        s, B = st["session"], c["B"]
        out = torch.zeros(B + NEW, dtype=torch.float64, device="cuda")
        pos = torch.cat([s.pos[:B], torch.arange(st["at"], st["at"] + NEW, device="cuda")])
        rows_pos = pos[-c["W"]:].repeat(c["Hq"] // c["H"])
        for l in range(c["M"]):
            k, v = (torch.cat([x[l, :, :B], y[l]], 1) for x, y in ((s.K, st["new"][0]), (s.V, st["new"][1])))
            rows, e = _row_stats(st["Q"][l].view(c["H"], -1, c["d"]), k, v, pos, rows_pos, torch.float64)
            out = torch.maximum(out, (e / rows[..., 1:2]).amax((0, 1)))
        return dict(scores=out, idx=None, k=None, v=None, pos=None, pages=None)
    trajs, lays, mask = _trajectories(c, seed), _layouts(c), _layers(c)
    if c["op"] in ("effects", "step"):
        pre = [_effects64(c, lay, t.K[:, :, :lay[0]], t.V[:, :, :lay[0]], t.Q_pre, t.pos[:lay[0]], t.qpos_pre, lay[4], mask)[0]
               for t, lay in zip(trajs, lays)]
        post = [_effects64(c, lay, t.K, t.V, t.Q_post, t.pos, t.qpos_post, len(lay[2]), mask) for t, lay in zip(trajs, lays)]
        out = dict(R_pre=pre, R_post=[r for r, _ in post], **_parts([s for _, s in post]))
        if c["op"] == "step":  # R_pre comes in a buffer of every page
            out["R_pre"] = [torch.cat([r, r.new_zeros(len(lay[2]) - lay[4])]) for r, lay in zip(pre, lays)]
            out.update({k: None for k in ("state", "cand", "n_cand", "accepted", "step_R", "idx", "n_idx", "k", "v", "pos")})
        return out
    if c["op"] == "from_stats":
        return dict(R_post=[_effects64(c, lay, t.K, t.V, t.Q_post, t.pos, t.qpos_post, len(lay[2]), mask)[0]
                            for t, lay in zip(trajs, lays)])
    if c["op"] == "tokens":
        outs = []
        for t in trajs:
            best = torch.zeros(t.pos.numel(), dtype=torch.float64, device="cuda")
            rows_pos = t.qpos_post.repeat(c["Hq"] // c["H"])
            for l in range(c["M"]):
                if mask and not mask[l]:
                    continue
                for h in range(c["H"]):
                    q = t.Q_post[l].view(c["H"], -1, c["d"])[h:h + 1]
                    st, e = _row_stats(q, t.K[l, h:h + 1], t.V[l, h:h + 1], t.pos, rows_pos, torch.float64)
                    best = torch.maximum(best, (e / st[..., 1:2]).amax((0, 1)))
            outs.append(best)
        return dict(scores=outs)
    st = prepare(c, seed)
    steps = []
    for t, lay, stats, cand, n in zip(st["trajs"], lays, st["stats"], st["cand"], st["n_cand"].tolist()):
        steps.append(_joint64(c, lay, t, stats, cand[:n].tolist(), mask))
    return dict(accepted=None, step_R=steps)
