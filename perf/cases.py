"""What is timed when the speed of this package is looked at: calls as a decoder makes them.

A case is a dict of plain sizes.  `prepare` makes on the GPU what such a decoder has in hand before
the call (caches, the step's projections and scores, the block's template, the context and the fork
sets), `run` makes the calls once, `work` counts the bytes and operations no implementation can do
without.  Kinds of cases:

  block    one or more blocks decoded by fdd_decode_block: per step, attention of every layer and
           unmasking, at the end of each block the append of its K/V.  The blocks join every
           rollout's private suffix or (extend) the shared prefix, by a fork set of one rollout that
           is made for them.  Afterwards the rollouts' trajectories are averaged (average "plain" or
           "jmt").
  cycle    one draft / verify cycle of Scaffold Speculative Decoding, call by call: bidirectional
           attention, drafts, causal attention, accept scan.
  attn     one attention call of a model whose own loop drives the layers.
  unmask   one unmasking call of such a loop, confidences asked for.
  host     one unmasking step whose scores lie in pinned host memory: rows pulled, then unmasked.

Scores follow the two shapes of the package's synthetic workloads: "peaked" (unit normal, one entry
raised so that its probability is sigmoid(m), m uniform in [0, 6]) and "flat" (normal, sigma 2: no
position is ever confident, each step commits one).
"""
import ctypes
import math
import random

import torch

from paper_2605_23163_b200 import fdd

N_INPUTS = 5                # score sets a block cycles through: most blocks are complete after four to six steps
WAYPOINTS = 10              # decoded waypoints per rollout
JMT_WAYPOINTS = 20          # waypoints after interpolation

BASE = dict(kind="block", hq=16, hkv=2, dim=128, prefix=4096, suffix=0, forks=8, block=32, scaffold=10, vocab=151936,
            logits="bf16", scores="peaked", threshold=0.9, temperature=1.0, page=0, layers=1, blocks=1, scenes=1,
            mix=0, extend=False, average="", causal=False)


def _case(**over):
    return dict(BASE, **over)


def listed():
    return [
        # The smallest block there is a workload for: one rollout, small head, fp32 scores that are never
        # confident, so a step per value position.  Nothing but latencies and launches.
        _case(name="block_small", hq=4, hkv=1, dim=64, prefix=256, forks=1, block=16, scaffold=4, vocab=4096, logits="f32",
              scores="flat", temperature=0.0),
        # The deterministic JSON sections: one greedy rollout whose blocks go to the shared prefix.
        _case(name="blocks_deterministic", forks=1, temperature=0.0, blocks=3, extend=True),
        # The trajectory section of one scene with the usual number of sampled rollouts.
        _case(name="blocks_rollouts", blocks=3, average="jmt"),
        # A block of the same with all layers of a small backbone and a ragged prefix.
        _case(name="block_rollouts_36_layers", prefix=4003, layers=36),
        # The largest single scene: long multi-camera context, many rollouts, long blocks.
        _case(name="block_long_prefix", hq=32, hkv=8, prefix=16384, forks=32, block=64, scaffold=26, threshold=0.8,
              average="plain"),
        # A server's batch: sixteen scenes of all sizes with paged prefixes in one call.
        _case(name="block_serving_mix", page=64, scenes=16, mix=5),
        # A backbone whose query heads come in groups of seven, ragged sizes.
        _case(name="block_group_of_7", hq=28, hkv=4, prefix=3001, forks=6, block=27, scaffold=8, layers=2),
        # Scaffold Speculative Decoding, one cycle driven call by call.
        _case(name="speculative_cycle", kind="cycle", suffix=96),
        # The model's own loop calls attention layer by layer: head dimension 64, ragged context and suffix.
        _case(name="attention_dim_64", kind="attn", hq=32, hkv=8, dim=64, prefix=8191, suffix=100, forks=16, block=48),
        # Scores kept in fp32, sampled below temperature 1.
        _case(name="unmask_fp32", kind="unmask", forks=16, block=64, scaffold=19, logits="f32", temperature=0.7),
        # A vocabulary that is not padded: rows start at any even address.
        _case(name="unmask_odd_vocabulary", kind="unmask", forks=12, block=48, scaffold=14, vocab=50257, temperature=0.0),
        # Scores produced elsewhere: they lie in pinned host memory.
        _case(name="host_scores", kind="host", forks=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["block", "block", "block", "cycle", "attn", "unmask", "host"])
    hq, hkv, dim = rng.choice([(4, 1, 64), (16, 2, 128), (16, 2, 128), (32, 8, 128), (32, 8, 64), (28, 4, 128), (12, 2, 128)])
    block = rng.randint(5, 64)
    c = _case(kind=kind, hq=hq, hkv=hkv, dim=dim, prefix=_log_int(rng, 100, 16384), forks=_log_int(rng, 1, 32),
              block=block, scaffold=int(block * rng.uniform(0.0, 0.5)),
              vocab=rng.choice([4096, 32000, 50257, 128256, 151936, 151936]), logits=rng.choice(["bf16", "bf16", "bf16", "f32"]),
              threshold=rng.choice([0.8, 0.9]), temperature=rng.choice([0.0, 0.7, 1.0, 1.0]), page=rng.choice([0, 0, 64]))
    if kind == "block":
        c["layers"], c["blocks"] = rng.choice([1, 1, 2, 4]), rng.choice([1, 1, 2, 3])
        if rng.random() < 0.25:
            c.update(scenes=rng.randint(2, 12), mix=rng.randint(1, 10**6), page=64, layers=1, blocks=1, hq=16, hkv=2, dim=128,
                     block=32, vocab=151936, logits="bf16")
            while sum(f * d for _, f, d, _ in _scenes(c)) > 4096:
                c["scenes"] -= 1
        elif c["forks"] == 1:
            c["extend"] = rng.random() < 0.5
        if c["vocab"] == 4096 and c["scenes"] == 1 and rng.random() < 0.5:
            c["scores"] = "flat"
        c["average"] = rng.choice(["", "plain", "jmt"]) if c["scenes"] == 1 else ""
    elif kind in ("attn", "cycle"):
        c["suffix"] = rng.choice([0, 0, rng.randint(1, 200)])
        c["causal"] = kind == "attn" and rng.random() < 0.3
    elif kind == "host":
        c["block"] = min(block, 48)
        c["scaffold"] = min(c["scaffold"], c["block"] // 2)
    # no dearer than the largest listed case, in scores as in attention (a group that is not a power of
    # two is held to what the other shapes take an eighth of the time for)
    esz = 2 if c["logits"] == "bf16" else 4
    while c["forks"] > 1 and c["scenes"] == 1:
        rows = c["forks"] * c["block"]
        keys = c["prefix"] + c["suffix"] + c["block"]
        g = c["hq"] // c["hkv"]
        pairs = rows * c["hq"] * keys * c["dim"] * c["layers"] * c["blocks"] * (64 if g & (g - 1) else 1)
        if rows * c["vocab"] * esz <= (64 << 20 if kind == "host" else 622329856) and pairs <= 2048 * 32 * 16448 * 128:
            break
        c["forks"] = (c["forks"] + 1) // 2
    return c


def _scenes(c):
    """(prefix, forks, block, scaffold) of every scene of the call."""
    if c["scenes"] == 1:
        return [(c["prefix"], c["forks"], c["block"], c["scaffold"])]
    r = random.Random(c["mix"])
    out = []
    for _ in range(c["scenes"]):
        d = r.choice([16, 32, 64])
        out.append((r.randint(2048, 12288), r.choice([1, 4, 16]), d, int(round(0.3 * d))))
    return out


class _Decoder:
    """A context and everything a case keeps alive; given back with the object."""

    ctx = None

    def __del__(self):
        if self.ctx is not None:
            fdd.fdd_destroy(self.ctx)
            self.ctx = None


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)


def _scores(c, rows, masked, gen):
    """Scores [rows, V]; only rows in `masked` (int64) carry values."""
    v = c["vocab"]
    out = torch.zeros((rows, v), dtype=torch.bfloat16 if c["logits"] == "bf16" else torch.float32, device="cuda")
    for at in range(0, len(masked), 256):
        idx = masked[at:at + 256]
        x = torch.randn((len(idx), v), generator=gen, device="cuda", dtype=torch.float32)
        if c["scores"] == "flat":
            x *= 2.0
        else:
            x = x.to(out.dtype).float()
            peak = torch.randint(0, v, (len(idx), 1), generator=gen, device="cuda")
            m = 6.0 * torch.rand((len(idx), 1), generator=gen, device="cuda")
            x.scatter_(1, peak, float("-inf"))
            x.scatter_(1, peak, torch.logsumexp(x, 1, keepdim=True) + m)
        out[idx] = x.to(out.dtype)
    return out


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    scenes = _scenes(c)
    hq, hkv, dim, layers, page = c["hq"], c["hkv"], c["dim"], c["layers"], c["page"]
    s = _Decoder()
    s.case = c
    s.forks = [x[1] for x in scenes]
    s.blocks = fdd.i32_array([x[2] for x in scenes])
    n = sum(s.forks)
    rows = sum(x[1] * x[2] for x in scenes)
    s.ctx = fdd.fdd_create(hq, hkv, dim, c["vocab"], layers, page, max(x[2] for x in scenes), n,
                           fdd.FDD_LOGITS_BF16 if c["logits"] == "bf16" else fdd.FDD_LOGITS_F32)
    s.scale = 1.0 / math.sqrt(dim)
    s.stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    # ---- the block's template: scaffold positions in place, the same for every rollout of a scene.
    # Tokens and states of the pass lie in one buffer, so that it starts with one copy.
    tokens, states = [], []
    for _, forks, d, scaffold in scenes:
        st = torch.zeros(d, dtype=torch.uint8, device="cuda")
        st[torch.randperm(d, generator=gen, device="cuda")[:scaffold]] = fdd.FDD_SCAFFOLD
        tk = torch.randint(0, c["vocab"] - 1, (d,), generator=gen, device="cuda", dtype=torch.int32)
        tk[st == fdd.FDD_MASKED] = c["vocab"] - 1
        tokens.append(tk.repeat(forks))
        states.append(st.repeat(forks))
    blocks = c["blocks"]
    s.template = torch.cat([torch.cat(tokens).repeat(blocks).view(torch.uint8), torch.cat(states).repeat(blocks)])
    s.work = s.template.clone()
    s.tokens = s.work[:4 * rows * blocks].view(torch.int32).view(blocks, rows)
    s.state = s.work[4 * rows * blocks:].view(blocks, rows)
    s.n_committed = torch.zeros(n, dtype=torch.int32, device="cuda")
    s.n_left = torch.zeros(n, dtype=torch.int32, device="cuda")
    masked = torch.nonzero(torch.cat(states) == fdd.FDD_MASKED).flatten()

    # ---- caches and fork sets
    s.fork_args, s.suffixes, s.keep = [], [], []
    for prefix, forks, d, _ in scenes:
        cap = prefix + (blocks * d if c["extend"] else 0)
        table = None
        if page:
            used = (cap + page - 1) // page
            cap = used + 3
            table = torch.randperm(cap, generator=gen, device="cuda")[:used].to(torch.int32)
            shape = (layers, cap, hkv, page, dim)
        else:
            shape = (layers, hkv, cap, dim)
        pk, pv = _normal(gen, *shape), _normal(gen, *shape)
        scap = c["suffix"] + blocks * d
        sk, sv = (torch.zeros((layers, forks, hkv, scap, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        seeds = fdd.u64_array([(seed * 1000003 + 7919 * len(s.fork_args) + f) for f in range(forks)])
        s.keep.append((pk, pv, table))
        s.suffixes.append((sk, sv))
        s.fork_args.append((fdd.ptr_array(list(pk)), fdd.ptr_array(list(pv)), table, prefix, cap, forks, seeds,
                            fdd.ptr_array(list(sk)), fdd.ptr_array(list(sv)), scap))
    s.sets = [] if c["extend"] else [fdd.fdd_fork(s.ctx, *a) for a in s.fork_args]
    s.sets_arr = fdd.ptr_array(s.sets)

    # ---- the step's projections (the model writes every step into the same buffers) and scores
    if c["kind"] in ("block", "cycle", "attn"):
        s.q = _normal(gen, layers, rows * hq * dim)
        s.k, s.v = _normal(gen, layers, rows * hkv * dim), _normal(gen, layers, rows * hkv * dim)
        s.out = torch.zeros((layers, rows * hq * dim), dtype=torch.bfloat16, device="cuda")
    if c["suffix"] and c["kind"] in ("block", "cycle", "attn"):
        # blocks committed earlier, of at most the context's block length each
        for at in range(0, c["suffix"], c["block"]):
            d = min(c["block"], c["suffix"] - at)
            for layer in range(layers):
                ek, ev = _normal(gen, n * d * hkv * dim), _normal(gen, n * d * hkv * dim)
                fdd.fdd_kv_commit(s.ctx, s.sets_arr, layer, ek, ev, [d], 1 if layer == layers - 1 else 0)
                s.keep.append((ek, ev))
    if c["kind"] == "block":
        s.scores = [_scores(c, rows, masked, gen) for _ in range(N_INPUTS)]
        steps = range(N_INPUTS)
        args = (layers, max(x[2] for x in scenes), fdd.ptr_array([t for _ in steps for t in s.q]),
                fdd.ptr_array([t for _ in steps for t in s.k]), fdd.ptr_array([t for _ in steps for t in s.v]),
                fdd.ptr_array([t for _ in steps for t in s.out]), fdd.ptr_array(s.scores))
        s.block_args = [(*args, s.tokens[b], s.state[b], s.blocks, s.scale, 0, c["threshold"], c["temperature"], b)
                        for b in range(blocks)]
        s.traj = 10.0 * torch.randn((n, WAYPOINTS, 2), generator=gen, device="cuda")
        s.traj_out = torch.zeros((JMT_WAYPOINTS if c["average"] == "jmt" else WAYPOINTS, 2), device="cuda")
        if not c["extend"]:
            s.calls = [fdd.decode_block_call(s.ctx, s.sets_arr, *a, 1, s.n_committed, s.n_left, stream=s.stream) for a in s.block_args]
    elif c["kind"] == "cycle":
        s.draft_scores, s.verify_scores = (_scores(c, rows, masked, gen) for _ in range(2))
        # the verifier agrees with most drafts: four rows in five have the same scores
        same = masked[torch.rand(len(masked), generator=gen, device="cuda") < 0.8]
        s.verify_scores[same] = s.draft_scores[same]
    elif c["kind"] in ("unmask", "host"):
        s.scores = _scores(c, rows, masked, gen)
        s.conf = torch.zeros(rows, dtype=torch.float32, device="cuda")
        if c["kind"] == "host":
            s.host = torch.empty(s.scores.shape, dtype=s.scores.dtype, pin_memory=True)
            s.host.copy_(s.scores)
            s.scores.zero_()
    return s


def _block(s):
    c = s.case
    s.work.copy_(s.template, non_blocking=True)
    if c["extend"]:
        # a set of one rollout made for these blocks: their K/V go behind the shared prefix
        sets = [fdd.fdd_fork(s.ctx, *a) for a in s.fork_args]
        for args in s.block_args:
            fdd.fdd_decode_block(s.ctx, sets, *args, 0, s.n_committed, s.n_left, stream=s.stream)
            for layer in range(c["layers"]):
                fdd.fdd_prefix_extend(s.ctx, sets, layer, s.k[layer], s.v[layer], s.blocks,
                                      1 if layer == c["layers"] - 1 else 0, stream=s.stream)
        for f in sets:
            fdd.fdd_forkset_free(s.ctx, f)
    else:
        for f in s.sets:
            fdd.fdd_forkset_reset(s.ctx, f)
        for call in s.calls:
            call()
    if c["average"] == "jmt":
        fdd.fdd_average_rollouts_jmt(s.ctx, s.traj, s.traj.shape[0], WAYPOINTS, JMT_WAYPOINTS, s.traj_out, stream=s.stream)
    elif c["average"]:
        fdd.fdd_average_rollouts(s.ctx, s.traj, s.traj.shape[0], WAYPOINTS, s.traj_out, stream=s.stream)
    caches = [t for pair in (s.suffixes if not c["extend"] else [x[:2] for x in s.keep[:1]]) for t in pair]
    return {"tokens": s.tokens, "state": s.state, "left": s.n_left, "out": s.out, "caches": caches, "trajectory": s.traj_out}


def run(s):
    c = s.case
    if c["kind"] == "block":
        return _block(s)
    if c["kind"] == "attn":
        fdd.fdd_block_attn(s.ctx, s.sets_arr, 0, s.q, s.k, s.v, s.out, s.blocks, s.scale, int(c["causal"]), stream=s.stream)
        return s.out
    s.work.copy_(s.template, non_blocking=True)
    if c["kind"] == "cycle":
        fdd.fdd_block_attn(s.ctx, s.sets_arr, 0, s.q, s.k, s.v, s.out, s.blocks, s.scale, 0, stream=s.stream)
        fdd.fdd_ss_draft(s.ctx, s.sets_arr, s.draft_scores, s.tokens, s.state, s.blocks, c["temperature"], 0, 0, s.n_committed,
                         s.n_left, stream=s.stream)
        fdd.fdd_block_attn(s.ctx, s.sets_arr, 0, s.q, s.k, s.v, s.out, s.blocks, s.scale, 1, stream=s.stream)
        fdd.fdd_ss_accept(s.ctx, s.sets_arr, s.verify_scores, s.tokens, s.state, s.blocks, c["temperature"], 0, 0, s.n_committed,
                          s.n_left, stream=s.stream)
        return {"tokens": s.tokens, "state": s.state, "accepted": s.n_committed, "left": s.n_left, "out": s.out}
    if c["kind"] == "host":
        fdd.fdd_pull_masked_rows(s.ctx, s.host, s.scores, s.state, None, stream=s.stream)
    fdd.fdd_unmask(s.ctx, s.sets_arr, s.scores, s.tokens, s.state, s.blocks, c["threshold"], c["temperature"], 0, 0,
                   s.n_committed, s.n_left, s.conf, stream=s.stream)
    return {"tokens": s.tokens, "state": s.state, "committed": s.n_committed, "left": s.n_left, "conf": s.conf}


def _commit_rate(c):
    """Expected share of the MASKED positions that a step commits ("peaked" scores)."""
    lt = math.log(c["threshold"] / (1.0 - c["threshold"]))
    if c["temperature"] == 0.0:
        return 1.0 - lt / 6.0
    return (math.log1p(math.exp(6.0)) - math.log1p(math.exp(lt))) / 6.0


def work(case):
    """Bytes and operations of one pass; where the number of steps depends on the scores, what is expected of it."""
    c = case
    esz = 2 if c["logits"] == "bf16" else 4
    hq, hkv, dim, layers = c["hq"], c["hkv"], c["dim"], c["layers"]
    total = {"bytes": 0.0, "flops": 0.0}

    def attention(prefix, suffix, forks, d, share=1.0):
        n = forks * share                                          # rollouts that take part
        any_on = 1.0 - (1.0 - share) ** forks                      # whether the shared prefix is read at all
        keys = prefix + suffix + d
        total["flops"] += layers * 4.0 * n * d * hq * keys * dim
        total["bytes"] += layers * 2.0 * dim * (2 * hkv * prefix * any_on + 2 * n * (suffix + d) * hkv + 2 * n * d * hq)

    def scores(rows):
        total["bytes"] += rows * c["vocab"] * esz
        total["flops"] += 4.0 * rows * c["vocab"]                  # compare, scale and subtract, exponential, sum

    for prefix, forks, d, scaffold in _scenes(c):
        value = d - scaffold
        if c["kind"] == "attn":
            attention(prefix, c["suffix"], forks, d)
        elif c["kind"] == "cycle":
            for _ in range(2):
                attention(prefix, c["suffix"], forks, d)
                scores(forks * value)
        elif c["kind"] in ("unmask", "host"):
            scores(forks * value)
        else:
            q = 1.0 - _commit_rate(c)
            steps = value if c["scores"] == "flat" else max(1, math.ceil(math.log(0.5 / max(1, forks * value)) / math.log(q)))
            for b in range(c["blocks"]):
                for t in range(steps):
                    left = value - t if c["scores"] == "flat" else value * q ** t
                    alive = 1.0 if c["scores"] == "flat" else 1.0 - (1.0 - q ** t) ** value
                    attention(prefix + (b * d if c["extend"] else 0), 0 if c["extend"] else b * d, forks, d, alive)
                    scores(forks * left)
                total["bytes"] += layers * 2 * 2 * 2.0 * forks * d * hkv * dim  # K and V of the block, read and written
    return total


def tolerance(case):
    c = case
    if c["kind"] in ("unmask", "host"):
        # fp32 sums of up to 152k exponentials: 4.4e-7 (largest 1.3e-6) against the same sums in 64 bits
        return {"rel": 2e-6, "max": 1e-5, "differ": 2e-3}
    # bf16 outputs of sums whose weights are rounded to bf16: 2.3e-3 (largest 0.011) against 64 bits
    return {"rel": 1e-2, "max": 0.05, "differ": 2e-3}


# ---- the same outputs in 64 bits, from the inputs alone
def _prefix(pk, table, layer, length):
    """Keys (or values) of the shared prefix, [length, hkv, dim]."""
    x = pk[layer]
    if table is None:
        return x[:, :length].transpose(0, 1)
    return x[table.long()].transpose(1, 2).flatten(0, 1)[:length]   # [pages, hkv, 64, dim] in the order of the table


def _attention64(q, k, v, scale, causal_from):
    """q [d, hq, dim] against k, v [keys, hkv, dim]; keys from causal_from on are visible up to the query's position."""
    d, hq, dim = q.shape
    hkv = k.shape[1]
    qh = q.view(d, hkv, hq // hkv, dim).permute(1, 2, 0, 3).reshape(hkv, -1, dim)
    sc = torch.matmul(qh, k.permute(1, 2, 0)) * scale
    if causal_from is not None:
        hidden = torch.ones((d, d), dtype=torch.bool, device=q.device).triu(1).repeat(hq // hkv, 1)
        sc[:, :, causal_from:].masked_fill_(hidden, float("-inf"))
    o = torch.matmul(torch.softmax(sc, -1), v.transpose(0, 1))
    return o.view(hkv, hq // hkv, d, dim).permute(2, 0, 1, 3).reshape(-1)


def _exact_attention(s):
    c = s.case
    hq, hkv, dim, causal = c["hq"], c["hkv"], c["dim"], c["causal"] or c["kind"] == "cycle"
    before = c["blocks"] - 1 if c["kind"] == "block" else 0          # blocks that join the caches ahead of the last one
    out = torch.zeros(s.out.shape, dtype=torch.float64, device="cuda")
    for layer in range(c["layers"]):
        at = 0
        for (prefix, forks, d, _), (pk, pv, table) in zip(_scenes(c), s.keep):
            shared = [_prefix(x, table, layer, prefix).double() for x in (pk, pv)]
            for f in range(forks):
                own = [x[layer].view(-1, hkv, dim)[at:at + d].double() for x in (s.k, s.v)]
                kv = [[shared[i]] + [own[i]] * before for i in range(2)]
                for e in s.keep[len(_scenes(c)):]:                   # blocks committed earlier (such cases have one scene and layer)
                    for i in range(2):
                        kv[i].append(e[i].view(forks, -1, hkv, dim)[f].double())
                k, v = (torch.cat(kv[i] + [own[i]]) for i in range(2))
                q = s.q[layer].view(-1, hq, dim)[at:at + d].double()
                out[layer, at * hq * dim:(at + d) * hq * dim] = _attention64(q, k, v, s.scale, len(k) - d if causal else None)
                at += d
    return out


def _exact_caches(s):
    c = s.case
    res, at = [], 0
    for (prefix, forks, d, _), (sk, sv), (pk, pv, table) in zip(_scenes(c), s.suffixes, s.keep):
        blocks = [x.view(c["layers"], -1, c["hkv"], c["dim"])[:, at:at + forks * d].view(c["layers"], forks, d, c["hkv"], c["dim"])
                  for x in (s.k, s.v)]
        at += forks * d
        if not c["extend"]:
            res += [b.transpose(2, 3).repeat(1, 1, 1, c["blocks"], 1).double() for b in blocks]
            continue
        pos = torch.arange(prefix, prefix + c["blocks"] * d, device="cuda")
        for cache, b in zip((pk, pv), blocks):
            x, rows = cache.double(), b[:, 0].repeat(1, c["blocks"], 1, 1).double()
            if table is None:
                x[:, :, pos] = rows.transpose(1, 2)
            else:
                x[:, table.long()[pos // c["page"]], :, pos % c["page"]] = rows.transpose(0, 1)
            res.append(x)
    return res


def _exact_trajectory(s):
    if not s.case["average"]:
        return torch.zeros(s.traj_out.shape, dtype=torch.float64, device="cuda")
    mean = s.traj.double().mean(0)
    if s.case["average"] == "plain":
        return mean
    # least integral of squared jerk through the origin and the waypoints: sums of |t - knot|^5 and a parabola
    n = WAYPOINTS + 1
    kt = torch.arange(n, dtype=torch.float64)
    par = torch.stack([kt ** e for e in range(3)], 1)
    lhs = torch.zeros((n + 3, n + 3), dtype=torch.float64)
    lhs[:n, :n], lhs[:n, n:], lhs[n:, :n] = (kt[:, None] - kt).abs() ** 5, par, par.T
    rhs = torch.zeros((n + 3, 2), dtype=torch.float64)
    rhs[1:n] = mean.cpu()
    w = torch.linalg.solve(lhs, rhs)
    t = (torch.arange(JMT_WAYPOINTS, dtype=torch.float64) + 1) * WAYPOINTS / JMT_WAYPOINTS
    return (torch.cat([(t[:, None] - kt).abs() ** 5, torch.stack([t ** e for e in range(3)], 1)], 1) @ w).cuda()


def _philox(c0, c1, key):
    """Philox4x32-10 of the counters (c0, c1, 0, 0): int64 tensors holding 32-bit words; four words in the last dimension."""
    low = 0xFFFFFFFF
    c = [c0, c1, torch.zeros_like(c0), torch.zeros_like(c0)]
    k = [key & low, key >> 32]
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]                # (wraps modulo 2^64: the same bits)
        c = [((p1 >> 32) & low) ^ c[1] ^ k[0], p1 & low, ((p0 >> 32) & low) ^ c[3] ^ k[1], p0 & low]
        k = [(k[0] + 0x9E3779B9) & low, (k[1] + 0xBB67AE85) & low]
    return torch.stack(c, -1)


def _gumbel(v, pos, keys):
    """Draws of rows with positions pos and seeds keys (int64, one per row) at step 0 of block 0, [rows, v]: an
    exponential race over groups of 16 ids whose leader the group's word names."""
    groups = (v + 15) // 16
    pos, keys = pos[:, None], keys[:, None]
    r = _philox(torch.arange((groups + 3) // 4, device="cuda") + 0 * pos, 0 * keys + pos, keys).flatten(1)[:, :groups]
    f = (_philox(torch.arange(groups * 4, device="cuda") + 0 * pos, 0 * keys + pos + 2 ** 31, keys) >> 9).view(len(pos), groups, 16)
    fine = (f.double() + 0.5) * 2.0 ** -23
    lead = (r & 15)[..., None]
    e_lead = -torch.log(((r >> 4).double()[..., None] + fine.gather(2, lead)) * 2.0 ** -28) / 16
    e = (e_lead - torch.log(fine)).scatter(2, lead, e_lead)
    return -torch.log(e).flatten(1)[:, :v]


def _exact_confidence(s, seed):
    c = s.case
    d, v = c["block"], c["vocab"]
    scores = s.host.cuda() if c["kind"] == "host" else s.scores
    conf = torch.full((c["forks"] * d,), float("nan"), dtype=torch.float64, device="cuda")
    masked = torch.nonzero(s.template[4 * len(conf):] == fdd.FDD_MASKED).flatten()
    for idx in masked.split(32):
        x = scores[idx].double()
        y = x if c["temperature"] == 0.0 else x + c["temperature"] * _gumbel(v, idx % d, seed * 1000003 + idx // d)
        conf[idx] = torch.exp(x.gather(1, y.argmax(1, keepdim=True))[:, 0] - torch.logsumexp(x, 1))
    return conf


def exact(case, seed):
    """What `run` returns, in 64 bits; whole numbers are left out."""
    c = case
    s = prepare(case, seed)
    if c["kind"] == "attn":
        return _exact_attention(s)
    if c["kind"] == "cycle":
        return {"tokens": None, "state": None, "accepted": None, "left": None, "out": _exact_attention(s)}
    if c["kind"] in ("unmask", "host"):
        return {"tokens": None, "state": None, "committed": None, "left": None, "conf": _exact_confidence(s, seed)}
    return {"tokens": None, "state": None, "left": None, "out": _exact_attention(s), "caches": _exact_caches(s),
            "trajectory": _exact_trajectory(s)}
