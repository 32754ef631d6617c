"""The work that a program using libedp has it do, as cases that can be timed.

Every case goes through the public entry points of paper_2609_24456_gb300.edp,
with the objects such a program keeps (a ring and its context, the batch
buffers, a captured graph) made in prepare().  Five families:

* stack  -- off-policy replay of single-channel frames: insertion, uniform or
            prioritized sampling, frame-stack delivery, priority update;
* mm     -- replay of normalised images with tokens, in one tier or two;
* ppo    -- one on-policy iteration: insertion of the rollout, advantages,
            shuffle, mini-batch deliveries;
* gae    -- advantages and returns alone;
* llm    -- group-relative advantages and packed delivery of token sequences.

Inputs come from the seed alone; the distributions are those of the
repository's fixtures (uniform bytes, rewards in {-1, 0, 1} or N(0, 1),
Exp(1) TD errors, Bernoulli episode ends, uniform response lengths).
"""
import math

import numpy as np
import torch

from paper_2609_24456_gb300 import edp

ALPHA, EPS, BETA = 0.6, 1e-6, 0.4        # prioritized replay
GAMMA, LAMBDA = 0.99, 0.95               # advantages
GRPO_EPS = 1e-6
MEAN, STD = (0.485, 0.456, 0.406, 0.45), (0.229, 0.224, 0.225, 0.226)


def listed():
    return [
        # the smallest call in earnest: a 10,000-frame replay that gets four
        # new transitions and delivers 32 stacks between two learner steps
        dict(name="dqn_b32", kind="stack", cap=10_000, h=84, w=84, stack=4, next_obs=True,
             prioritized=False, batch=32, ingest=4, rounds=0),
        # prioritized replay at its usual size, four learner rounds per
        # replay of a captured graph
        dict(name="per_1m_b512", kind="stack", cap=1_000_000, h=84, w=84, stack=4,
             next_obs=True, prioritized=True, batch=512, ingest=0, rounds=4),
        # small observations (128 bytes) in a large batch: many actors insert,
        # one learner takes 32,768 transitions and returns their priorities
        dict(name="per_vec_b32768", kind="stack", cap=1_000_000, h=8, w=16, stack=1,
             next_obs=True, prioritized=True, batch=32_768, ingest=4_096, rounds=0),
        # a frame side and a batch that divide nothing evenly, three frames,
        # no successor
        dict(name="stack_92_b1021", kind="stack", cap=100_000, h=92, w=92, stack=3,
             next_obs=False, prioritized=False, batch=1021, ingest=0, rounds=0),
        # images with tokens, the batch of the repository's benchmark
        dict(name="mm_b1024", kind="mm", cap=20_000, cap_h=20_000, c=3, h=224, w=224,
             tokens=512, batch=1024, ingest=0),
        # a ring of two tiers: insertion demotes, delivery reads both
        dict(name="mm_tier_b128", kind="mm", cap=4_096, cap_h=2_048, c=3, h=96, w=96,
             tokens=128, batch=128, ingest=64),
        # the on-policy iteration of the repository's benchmark
        dict(name="ppo_img_256x128", kind="ppo", T=128, E=256, c=3, h=64, w=64, parts=8),
        # thousands of simulated environments with small observations
        dict(name="ppo_vec_4096x64", kind="ppo", T=64, E=4_096, c=1, h=8, w=16, parts=4),
        # few environments, long rollouts
        dict(name="gae_8x2048", kind="gae", T=2_048, E=8),
        # a whole post-training batch: advantages and one packed delivery
        dict(name="grpo_512x16", kind="llm", prompts=512, group=16, lmin=128, lmax=4_096,
             batch=8_192, fused=True, values=True),
        # one learner micro-batch of long responses
        dict(name="pack_long_b64", kind="llm", prompts=64, group=8, lmin=2_048, lmax=32_768,
             batch=64, fused=False, values=True),
        # many short sequences
        dict(name="pack_short_b65536", kind="llm", prompts=16_384, group=8, lmin=8, lmax=256,
             batch=65_536, fused=False, values=True),
    ]


# --- draws ---------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_stack(rng):
    if rng.random() < 0.4:
        h, w = rng.choice([(8, 16), (16, 16), (4, 36)])
    else:
        h = w = 4 * rng.randint(4, 32)
    new = rng.choice([0, _log(rng, 1, 8_192)])
    most = (1 if new else 4) * 1_000_000_000 // (h * w)
    return dict(kind="stack", cap=_log(rng, 10_000, min(1_000_000, most)), h=h, w=w,
                stack=rng.choice([1, 2, 3, 4, 4, 8]), next_obs=rng.random() < 0.6,
                prioritized=rng.random() < 0.6, batch=_log(rng, 16, 32_768), ingest=new,
                rounds=0)


def _draw_mm(rng):
    side = 4 * rng.randint(16, 64)
    c = rng.choice([1, 3, 3])
    cap = _log(rng, 2_000, 20_000)
    tier = rng.random() < 0.3
    if tier:
        cap = min(cap, 400_000_000 // (c * side * side))
    return dict(kind="mm", cap=cap, cap_h=cap // 2 + 1 if tier else cap, c=c, h=side, w=side,
                tokens=4 * rng.choice([0, 1, rng.randint(2, 256)]),
                batch=_log(rng, 8, 200 if tier else 1024),
                ingest=_log(rng, 1, 64) if tier or rng.random() < 0.5 else 0)


def _draw_ppo(rng):
    E = _log(rng, 8, 4_096)
    T = _log(rng, 16, max(17, min(1_024, 262_144 // E)))
    h, w = rng.choice([(8, 16), (16, 16), (32, 32), (36, 28), (64, 64)])
    return dict(kind="ppo", T=T, E=E, c=rng.randint(1, 4), h=h, w=w,
                parts=rng.choice([1, 2, 4, 5, 8, 16]))


def _draw_gae(rng):
    E = _log(rng, 1, 8_192)
    return dict(kind="gae", T=_log(rng, 8, min(8_192, 2_000_000 // E)), E=E)


def _draw_llm(rng):
    lmax = _log(rng, 32, 32_768)
    group = rng.choice([4, 7, 8, 16, 64])
    prompts = max(1, min(_log(rng, 8, 16_384), 17_000_000 // (lmax * group)))
    fused = rng.random() < 0.5
    n = prompts * group
    return dict(kind="llm", prompts=prompts, group=group, lmin=rng.choice([0, 1, lmax // 8]),
                lmax=lmax, batch=n if fused else min(n, _log(rng, 1, n)), fused=fused,
                values=fused or rng.random() < 0.7)


def draw(rng):
    most = max(work(c)["bytes"] for c in listed())
    while True:
        c = rng.choice([_draw_stack, _draw_stack, _draw_mm, _draw_ppo, _draw_gae,
                        _draw_llm])(rng)
        if work(c)["bytes"] <= most:
            return c


# --- inputs ----------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _bytes(g, rows, row):
    n = -(-rows * row // 8)
    x = torch.empty(n, dtype=torch.int64, device="cuda")
    x.random_(-(1 << 63), None, generator=g)
    return x.view(torch.uint8)[:rows * row].view(rows, row)


def _meta(g, n, done_p=0.01):
    action = torch.randint(0, 6, (n,), generator=g, device="cuda", dtype=torch.int32)
    u = torch.rand(n, generator=g, device="cuda")
    reward = (u > 0.9).float() - (u < 0.1).float()
    done = (torch.rand(n, generator=g, device="cuda") < done_p).to(torch.uint8)
    return action, reward, done


def _exp1(g, *shape):
    return torch.empty(shape, device="cuda").exponential_(1.0, generator=g)


def _stack_inputs(c, seed):
    """What the ring is filled with (more transitions than it holds, so that
    it has wrapped), what is inserted in a pass, and the TD errors."""
    g = _gen(seed)
    F, total = c["h"] * c["w"], c["cap"] + c["cap"] // 8 + 5
    fill = (_bytes(g, total, F),) + _meta(g, total)
    q = None
    if c["prioritized"]:
        q = ((_exp1(g, total) + EPS).pow(ALPHA) * 2**20).to(torch.int32).clamp_(min=1)
    new = ((_bytes(g, c["ingest"], F),) + _meta(g, c["ingest"])) if c["ingest"] else None
    td = _exp1(g, 1 + c["rounds"], c["batch"]) if c["prioritized"] else None
    return fill, q, new, td


def _mm_inputs(c, seed):
    g = _gen(seed)
    row, total = c["c"] * c["h"] * c["w"], c["cap"] + c["cap"] // 8 + 5

    def rows(n):
        tok = (torch.randint(0, 32_000, (n, c["tokens"]), generator=g, device="cuda",
                             dtype=torch.int32) if c["tokens"] else None)
        return _bytes(g, n, row), tok, torch.randn(n, generator=g, device="cuda")

    return rows(total), rows(c["ingest"]) if c["ingest"] else None


def _rollout(g, T, E, done_p=0.005):
    r = torch.randn(T, E, generator=g, device="cuda")
    v = torch.randn(T + 1, E, generator=g, device="cuda")
    d = (torch.rand(T, E, generator=g, device="cuda") < done_p).to(torch.uint8)
    return r, v, d


def _ppo_inputs(c, seed):
    g = _gen(seed)
    return _bytes(g, c["T"] * c["E"], c["c"] * c["h"] * c["w"]), _rollout(g, c["T"], c["E"])


def _llm_inputs(c, seed):
    """Token array, offsets, rewards (0/1 for half of the groups, N(0, 1) for
    the others) and the order in which the batch takes the sequences."""
    g = _gen(seed)
    n = c["prompts"] * c["group"]
    lens = torch.randint(c["lmin"], c["lmax"] + 1, (n,), generator=g, device="cuda")
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    tokens = torch.randint(0, 152_064, (int(off[-1]),), generator=g, device="cuda",
                           dtype=torch.int32)
    binary = (torch.rand(c["prompts"], generator=g, device="cuda") < 0.5).repeat_interleave(
        c["group"])
    r = torch.where(binary, (torch.rand(n, generator=g, device="cuda") < 0.4).float(),
                    torch.randn(n, generator=g, device="cuda"))
    idx = torch.randperm(n, generator=g, device="cuda")[:c["batch"]].contiguous()
    goff = torch.arange(0, n + 1, c["group"], dtype=torch.int64, device="cuda")
    return tokens, off, lens, r, goff, idx


# --- prepare ---------------------------------------------------------------------
class _DeviceArray:
    """n int32 of a ring's memory at a device address, for torch.as_tensor (no
    copy); the tensor keeps the ring."""

    def __init__(self, ring, p, n):
        self.ring = ring
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i4", "data": (p, False),
                                         "version": 2}


def _ingest_all(ring, obs, q=None, **fields):
    """The whole fill, at most a ring's capacity at a time."""
    n, cap = obs.shape[0], ring.cfg.capacity
    for lo in range(0, n, cap):
        hi = min(n, lo + cap)
        part = {k: v[lo:hi].clone() if v is not None else None for k, v in fields.items()}
        edp.edp_ingest(ring.ctx, obs[lo:hi].clone(), hi - lo,
                       q=None if q is None else q[lo:hi].clone(), **part)
    torch.cuda.synchronize()


def _stack_outputs(c):
    B, K, h, w = c["batch"], c["stack"], c["h"], c["w"]
    dev = dict(device="cuda")
    o = dict(idx=torch.zeros(B, dtype=torch.int64, **dev),
             obs=torch.zeros(B, K, h, w, **dev),
             action=torch.zeros(B, dtype=torch.int32, **dev),
             reward=torch.zeros(B, **dev), done=torch.zeros(B, dtype=torch.uint8, **dev))
    if c["next_obs"]:
        o["next_obs"] = torch.zeros(B, K, h, w, **dev)
    if c["prioritized"]:
        o["q"] = torch.zeros(B, dtype=torch.int32, **dev)
        o["isw"] = torch.zeros(B, **dev)
    batch = edp.make_batch(o["obs"], o.get("next_obs"), o["action"], o["reward"], o["done"],
                           q=o.get("q"), isw=o.get("isw"), beta=BETA)
    return o, batch


def _stack_round(s, k, o, batch):
    """One learner round: draw, deliver, return the new priorities."""
    c, ctx = s["case"], s["ring"].ctx
    if c["prioritized"]:
        edp.edp_sample(ctx, edp.EDP_SAMPLE_PRIORITIZED, c["batch"], s["seed"], k, o["idx"],
                       o["q"])
        edp.edp_deliver(ctx, o["idx"], c["batch"], batch)
        edp.edp_update_priorities_td(ctx, o["idx"], s["td"][k % s["td"].shape[0]], c["batch"],
                                     ALPHA, EPS)
    else:
        edp.edp_sample_deliver(ctx, c["batch"], s["seed"], k, o["idx"], batch)


def _prepare_stack(c, seed):
    (obs, action, reward, done), q, new, td = _stack_inputs(c, seed)
    cfg = edp.make_config(c["cap"], (1, c["h"], c["w"]), edp.EDP_XFORM_STACK_F32,
                          frame_stack=c["stack"], next_obs=c["next_obs"],
                          prioritized=c["prioritized"])
    ring = edp.Ring(cfg)
    _ingest_all(ring, obs, q, action=action, reward=reward, done=done)
    s = dict(case=c, seed=int(seed), ring=ring, new=new, td=td, round=0)
    o, batch = _stack_outputs(c)
    s["out"] = o
    s["batch"] = batch
    s["state"] = {}
    if c["prioritized"]:
        s["state"]["leaves"] = torch.as_tensor(
            _DeviceArray(ring, ring.info().tree_leaves, c["cap"]), device="cuda")
    if c["ingest"]:
        s["state"].update(ring_obs=ring.obs, ring_action=ring.action, ring_reward=ring.reward,
                          ring_done=ring.done)
    if c["rounds"]:
        _stack_round(s, 0, o, batch)  # before the capture, as a program would
        s["outs"] = [_stack_outputs(c) for _ in range(c["rounds"])]
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], capture_error_mode="thread_local"):
            for k, (ok, bk) in enumerate(s["outs"]):
                _stack_round(s, 1 + k, ok, bk)
    return s


def _prepare_mm(c, seed):
    (obs, tok, rew), new = _mm_inputs(c, seed)
    cfg = edp.make_config(c["cap"], (c["c"], c["h"], c["w"]), edp.EDP_XFORM_CHW_NORM_BF16,
                          hbm_capacity=c["cap_h"], tokens=c["tokens"], norm_mean=MEAN,
                          norm_std=STD)
    ring = edp.Ring(cfg, action=False, done=False)
    _ingest_all(ring, obs, tokens=tok, reward=rew)
    B = c["batch"]
    o = dict(idx=torch.zeros(B, dtype=torch.int64, device="cuda"),
             obs=torch.zeros(B, c["c"], c["h"], c["w"], dtype=torch.bfloat16, device="cuda"),
             reward=torch.zeros(B, device="cuda"))
    if c["tokens"]:
        o["tokens"] = torch.zeros(B, c["tokens"], dtype=torch.int32, device="cuda")
    batch = edp.make_batch(o["obs"], reward=o["reward"], tokens=o.get("tokens"))
    s = dict(case=c, seed=int(seed), ring=ring, new=new, out=o, batch=batch, round=0, state={})
    if c["ingest"]:
        s["state"] = {k: v for k, v in dict(
            ring_obs=ring.obs, ring_tokens=ring.tokens, ring_reward=ring.reward,
            host_obs=ring.host_obs, host_tokens=ring.host_tokens).items() if v is not None}
    return s


def _prepare_ppo(c, seed):
    obs, (r, v, d) = _ppo_inputs(c, seed)
    n = c["T"] * c["E"]
    cfg = edp.make_config(n, (c["c"], c["h"], c["w"]), edp.EDP_XFORM_HWC_CHW_BF16)
    ring = edp.Ring(cfg, action=False, reward=False, done=False)
    f = lambda *sh: torch.zeros(sh, device="cuda")  # noqa: E731
    o = dict(adv=f(c["T"], c["E"]), ret=f(c["T"], c["E"]), adv_norm=f(c["T"], c["E"]),
             idx=torch.zeros(n, dtype=torch.int64, device="cuda"),
             obs=torch.zeros(n, c["c"], c["h"], c["w"], dtype=torch.bfloat16, device="cuda"),
             mb_adv=f(n), mb_ret=f(n))
    cuts = [n * m // c["parts"] for m in range(c["parts"] + 1)]
    parts = []
    for lo, hi in zip(cuts, cuts[1:]):
        if hi > lo:
            parts.append((o["idx"][lo:hi], hi - lo, edp.make_batch(
                o["obs"][lo:hi], gather=[(o["adv_norm"], o["mb_adv"][lo:hi]),
                                         (o["ret"], o["mb_ret"][lo:hi])])))
    return dict(case=c, seed=int(seed), ring=ring, obs=obs, rollout=(r, v, d), out=o,
                parts=parts, round=0)


def _small_ring():
    """A context that only names the GPU (advantages and packing use no ring)."""
    return edp.Ring(edp.make_config(16, (1, 4, 4), edp.EDP_XFORM_CHW_NORM_BF16), action=False,
                    reward=False, done=False)


def _prepare_gae(c, seed):
    r, v, d = _rollout(_gen(seed), c["T"], c["E"])
    o = {k: torch.zeros(c["T"], c["E"], device="cuda") for k in ("adv", "ret", "adv_norm")}
    return dict(case=c, ring=_small_ring(), rollout=(r, v, d), out=o)


def _prepare_llm(c, seed):
    tokens, off, lens, r, goff, idx = _llm_inputs(c, seed)
    # buffers for the longest batch there can be; what a batch leaves is 0
    n, room = c["prompts"] * c["group"], c["batch"] * c["lmax"]
    o = dict(tokens=torch.zeros(room, dtype=torch.int32, device="cuda"),
             off=torch.zeros(c["batch"] + 1, dtype=torch.int64, device="cuda"))
    if c["values"]:
        o["value"] = torch.zeros(room, device="cuda")
    if c["fused"]:
        o["adv"] = torch.zeros(n, device="cuda")
    return dict(case=c, ring=_small_ring(), tokens=tokens, seq_off=off, r=r, goff=goff, idx=idx,
                n=n, room=room, out=o)


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


# --- run -------------------------------------------------------------------------
def _run_stack(s):
    c, ring, k = s["case"], s["ring"], s["round"]
    if c["rounds"]:
        s["graph"].replay()
        return dict(rounds=[o for o, _ in s["outs"]], **s["state"])
    if s["new"] is not None:
        obs, action, reward, done = s["new"]
        edp.edp_ingest(ring.ctx, obs, c["ingest"], action=action, reward=reward, done=done)
    _stack_round(s, k, s["out"], s["batch"])
    s["round"] = k + 1
    return dict(s["out"], **s["state"])


def _run_mm(s):
    c, ring, k = s["case"], s["ring"], s["round"]
    if s["new"] is not None:
        obs, tok, rew = s["new"]
        edp.edp_ingest(ring.ctx, obs, c["ingest"], tokens=tok, reward=rew)
    edp.edp_sample_deliver(ring.ctx, c["batch"], s["seed"], k, s["out"]["idx"], s["batch"])
    s["round"] = k + 1
    return dict(s["out"], **s["state"])


def _run_ppo(s):
    c, ctx, o, k = s["case"], s["ring"].ctx, s["out"], s["round"]
    n = c["T"] * c["E"]
    edp.edp_ingest(ctx, s["obs"], n)
    edp.edp_gae(ctx, *s["rollout"], c["T"], c["E"], GAMMA, LAMBDA, adv=o["adv"], ret=o["ret"],
                adv_norm=o["adv_norm"])
    edp.edp_sample(ctx, edp.EDP_SAMPLE_PERMUTE, n, s["seed"], k, o["idx"])
    for idx, m, batch in s["parts"]:
        edp.edp_deliver(ctx, idx, m, batch)
    s["round"] = k + 1
    return dict(o, ring_obs=s["ring"].obs)


def _run_gae(s):
    c, o = s["case"], s["out"]
    edp.edp_gae(s["ring"].ctx, *s["rollout"], c["T"], c["E"], GAMMA, LAMBDA, adv=o["adv"],
                ret=o["ret"], adv_norm=o["adv_norm"])
    return o


def _run_llm(s):
    c, o = s["case"], s["out"]
    if c["fused"]:
        edp.edp_grpo_pack_deliver(s["ring"].ctx, s["r"], s["goff"], c["prompts"], GRPO_EPS,
                                  o["adv"], s["tokens"], s["seq_off"], s["n"], s["idx"],
                                  c["batch"], o["tokens"], o["off"], s["room"],
                                  out_value=o["value"])
    else:
        edp.edp_pack_deliver(s["ring"].ctx, s["tokens"], s["seq_off"], s["n"], s["idx"],
                             c["batch"], o["tokens"], o["off"], s["room"],
                             seq_value=s["r"] if c["values"] else None,
                             out_value=o.get("value"))
    return o


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state)


# --- work ------------------------------------------------------------------------
def work(case):
    c = case
    if c["kind"] == "stack":
        F, K, B = c["h"] * c["w"], c["stack"], c["batch"]
        nxt, pr = int(c["next_obs"]), int(c["prioritized"])
        # frames read once, stacks written, scalars, index; priorities read
        # and weights written; TD errors read and leaves written
        per = (K + nxt) * F + 4 * K * F * (1 + nxt) + 18 + 8 + pr * (8 + 4 + 4 + 4)
        n = c["ingest"]
        return {"bytes": max(1, c["rounds"]) * B * per + n * (2 * F + 18 + 4 * pr), "flops": 0}
    if c["kind"] == "mm":
        row = c["c"] * c["h"] * c["w"]
        # an insertion into a full two-tier ring also moves as many rows down
        moved = 2 if c["cap_h"] == c["cap"] else 4
        per = 3 * row + 8 * c["tokens"] + 8 + 8
        return {"bytes": c["batch"] * per +
                c["ingest"] * (moved * (row + 4 * c["tokens"]) + 8), "flops": 0}
    if c["kind"] == "ppo":
        n, row = c["T"] * c["E"], c["c"] * c["h"] * c["w"]
        # rows in (read, written), advantages, order, rows out with two scalars
        return {"bytes": n * (2 * row + 21 + 8 + 3 * row + 8 + 16) + 4 * c["E"], "flops": 0}
    if c["kind"] == "gae":
        return {"bytes": 21 * c["T"] * c["E"] + 4 * c["E"], "flops": 0}
    tokens = c["batch"] * (c["lmin"] + c["lmax"]) / 2
    n = c["prompts"] * c["group"]
    return {"bytes": tokens * (12 if c["values"] else 8) + c["batch"] * 32 +
            (8 * n + 8 * c["prompts"] if c["fused"] else 4 * c["batch"] * c["values"]),
            "flops": 0}


# --- tolerance -------------------------------------------------------------------
def tolerance(case):
    # The gathers and byte transforms are defined to the last bit (one
    # correctly rounded binary32 division; bfloat16 rounded to nearest even),
    # so cases without another sum or power are exact.
    if case["kind"] == "mm" or (case["kind"] == "stack" and not case["prioritized"]):
        return "exact"
    if case["kind"] == "stack":
        # weights: a power rounded once to 32 bits; priorities: a power
        # rounded to a whole number, at times to its neighbour
        return {"rel": 2.5e-7, "max": 5e-7, "differ": 1e-5}
    # advantages: sums of at least 44 bits rounded once to 32 (6e-8), and the
    # normalised ones computed from the rounded
    return {"rel": 2.5e-7, "max": 1e-6}


# --- exact: the same in 64 bits, without the library ------------------------------
_M32 = np.uint64(0xFFFFFFFF)


def _philox(seed, j, rnd, stream):
    """Word pairs of Philox4x32-10 (Salmon et al., SC'11) as uint64."""
    u = np.uint64
    x = [j.astype(u), np.full(j.shape, rnd & 0xFFFFFFFF, u), np.full(j.shape, stream, u),
         np.full(j.shape, rnd >> 32, u)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        p0, p1 = u(0xD2511F53) * x[0], u(0xCD9E8D57) * x[2]
        x = [(p1 >> u(32)) ^ x[1] ^ u(k0), p1 & _M32, (p0 >> u(32)) ^ x[3] ^ u(k1), p0 & _M32]
    return (x[1] << u(32)) | x[0]


def _mulhi(a, n):
    """High words of a * n (uint64 arrays; n below 2^63)."""
    u = np.uint64
    n = np.broadcast_to(np.asarray(n, dtype=u), a.shape)
    ah, al, nh, nl = a >> u(32), a & _M32, n >> u(32), n & _M32
    mid = ah * nl + ((al * nl) >> u(32))
    mid2 = al * nh + (mid & _M32)
    return ah * nh + (mid >> u(32)) + (mid2 >> u(32))


class _Priorities:
    """Leaves by slot, the newest transition's deferred."""

    def __init__(self, cap, defer, q):
        self.cap, self.defer = cap, defer
        self.total, self.leaves = len(q), np.zeros(cap, np.int64)
        ids = np.arange(max(0, len(q) - cap), len(q))
        self.leaves[ids % cap] = q[ids]
        self.qmax = max(1 << 20, int(q.max()))
        if defer:
            self.pending = int(q[-1])
            self.leaves[(len(q) - 1) % cap] = 0

    def ingest(self, n):
        if self.defer:
            self.leaves[(self.total - 1) % self.cap] = self.pending
            self.pending = self.qmax
        self.leaves[(self.total + np.arange(n)) % self.cap] = self.qmax
        self.total += n
        if self.defer:
            self.leaves[(self.total - 1) % self.cap] = 0

    def sample(self, B, seed, rnd):
        cs = np.cumsum(self.leaves)
        S = int(cs[-1])
        edge = np.array([k * S // B for k in range(B + 1)], dtype=np.uint64)
        t = edge[:-1] + _mulhi(_philox(seed, np.arange(B), rnd, 1), edge[1:] - edge[:-1])
        idx = np.searchsorted(cs, t.astype(np.int64), side="right")
        return idx, self.leaves[idx]

    def update(self, idx, td):
        x = np.abs(td.astype(np.float64)) + EPS
        q = np.clip(np.rint(x**ALPHA * 2.0**20), 1, 2**32 - 1).astype(np.int64)
        self.qmax = max(self.qmax, int(q.max()))
        newest = (self.total - 1) % self.cap
        for i, v in zip(idx.tolist(), q.tolist()):
            if self.defer and i == newest:
                self.pending = v
            else:
                self.leaves[i] = v


def _stacks(c, frames, done, total, slots):
    """obs and next_obs of the sampled slots, frames and done by id."""
    cap, K = c["cap"], c["stack"]
    oldest = max(0, total - cap)
    anchor = oldest + (torch.as_tensor(slots, device="cuda") - oldest) % cap
    got = []
    for shift in ([0, 1] if c["next_obs"] else [0]):
        out = torch.zeros(len(anchor), K, frames.shape[1], dtype=torch.float64, device="cuda")
        for m in range(K):
            lid = anchor - (K - 1) + m + shift
            ok = lid >= oldest
            for back in range(K):
                # an episode end at an id from this frame to before the newest one
                at = lid + back
                inside = at < anchor + shift
                ok &= ~(inside & (done[at.clamp(min=0, max=total - 1)] != 0))
            x = frames[lid.clamp(min=0, max=total - 1)].double() / 255.0
            out[:, m] = torch.where(ok[:, None], x, torch.zeros((), dtype=torch.float64,
                                                               device="cuda"))
        got.append(out.view(-1, K, c["h"], c["w"]))
    return got


def _exact_stack(c, seed):
    (obs, action, reward, done), q, new, td = _stack_inputs(c, seed)
    if new is not None:
        obs, reward, done = (torch.cat([a, b]) for a, b in
                             zip((obs, reward, done), (new[0], new[2], new[3])))
    total, cap = obs.shape[0], c["cap"]
    seed, defer = int(seed), int(c["next_obs"])
    oldest = max(0, total - cap)

    def outputs(idx, q=None):
        st = _stacks(c, obs, done, total, idx)
        lid = oldest + (torch.as_tensor(idx, device="cuda") - oldest) % cap
        o = dict(obs=st[0], action=None, reward=reward[lid].double(), done=None, idx=None)
        if c["next_obs"]:
            o["next_obs"] = st[1]
        if q is not None:
            o.update(q=None, isw=torch.from_numpy((q.min() / q.astype(np.float64))**BETA))
        return o

    state = {}
    if c["ingest"]:
        by_slot = torch.zeros(cap, dtype=torch.float64, device="cuda")
        ids = torch.arange(oldest, total, device="cuda")
        by_slot[ids % cap] = reward[ids].double()
        state = dict(ring_obs=None, ring_action=None, ring_reward=by_slot, ring_done=None)
    if not c["prioritized"]:
        u = _philox(seed, np.arange(c["batch"]), 0, 0)
        off = _mulhi(u, np.uint64(cap - defer)).astype(np.int64)
        return dict(outputs((oldest + off) % cap), **state)
    p = _Priorities(cap, defer, q.cpu().numpy().astype(np.int64))
    if c["ingest"]:
        p.ingest(c["ingest"])
    td, rounds = td.cpu().numpy(), []
    for k in range(1 + c["rounds"]):
        idx, qk = p.sample(c["batch"], seed, k)
        if k or not c["rounds"]:
            rounds.append(outputs(idx, qk))
        p.update(idx, td[k])
    state["leaves"] = None
    return dict(rounds=rounds, **state) if c["rounds"] else dict(rounds[0], **state)


def _exact_mm(c, seed):
    (obs, tok, rew), new = _mm_inputs(c, seed)
    if new is not None:
        obs, rew = torch.cat([obs, new[0]]), torch.cat([rew, new[2]])
    total, cap = obs.shape[0], c["cap"]
    oldest = total - cap
    off = _mulhi(_philox(int(seed), np.arange(c["batch"]), 0, 0), np.uint64(cap))
    lid = torch.from_numpy(off.astype(np.int64)).cuda() + oldest
    # the constants are the 32-bit ones that the context is given
    m = torch.tensor(MEAN[:c["c"]]).cuda().double().view(1, -1, 1, 1)
    s = torch.tensor(STD[:c["c"]]).cuda().double().view(1, -1, 1, 1)
    x = obs[lid].view(-1, c["c"], c["h"], c["w"])
    o = dict(idx=None, obs=(x.double() / 255.0 - m) / s, reward=rew[lid].double())
    if c["tokens"]:
        o["tokens"] = None
    if c["ingest"]:
        by_slot = torch.zeros(cap, dtype=torch.float64, device="cuda")
        ids = torch.arange(oldest, total, device="cuda")
        by_slot[ids % cap] = rew[ids].double()
        o["ring_reward"] = by_slot
    return o


def _exact_gae_of(T, E, r, v, d):
    r, v, live = r.double(), v.double(), 1.0 - d.double()
    adv = torch.zeros(T, E, dtype=torch.float64, device="cuda")
    delta = r + GAMMA * v[1:] * live - v[:-1]
    a = torch.zeros(E, dtype=torch.float64, device="cuda")
    for t in range(T - 1, -1, -1):
        a = delta[t] + GAMMA * LAMBDA * live[t] * a
        adv[t] = a
    std = adv.std() if T * E > 1 else torch.zeros((), dtype=torch.float64, device="cuda")
    return dict(adv=adv, ret=adv + v[:-1], adv_norm=(adv - adv.mean()) / (std + 1e-8))


def _exact_gae(c, seed):
    return _exact_gae_of(c["T"], c["E"], *_rollout(_gen(seed), c["T"], c["E"]))


def _exact_ppo(c, seed):
    obs, roll = _ppo_inputs(c, seed)
    o = _exact_gae_of(c["T"], c["E"], *roll)
    key = _philox(int(seed), np.arange(c["T"] * c["E"]), 0, 2)
    order = torch.from_numpy(np.argsort(key, kind="stable")).cuda()
    x = obs[order].view(-1, c["h"], c["w"], c["c"]).permute(0, 3, 1, 2).contiguous()
    return dict(o, idx=None, obs=x.double() / 255.0, mb_adv=o["adv_norm"].view(-1)[order],
                mb_ret=o["ret"].view(-1)[order], ring_obs=None)


def _exact_llm(c, seed):
    tokens, off, lens, r, goff, idx = _llm_inputs(c, seed)
    o = dict(tokens=None, off=None)
    val = r.double()
    if c["fused"]:
        g = val.view(-1, c["group"])
        std = g.std(1, keepdim=True) if c["group"] > 1 else torch.zeros_like(g[:, :1])
        eps = float(np.float32(GRPO_EPS))
        val = o["adv"] = ((g - g.mean(1, keepdim=True)) / (std + eps)).view(-1)
    if c["values"]:
        v = val[idx].repeat_interleave(lens[idx])
        o["value"] = torch.zeros(c["batch"] * c["lmax"], dtype=torch.float64, device="cuda")
        o["value"][:len(v)] = v
    return o


def exact(case, seed):
    return globals()["_exact_" + case["kind"]](case, seed)
