"""GPU parity of the scene-level paths: several layers with caches of their own, the order of
Sec. 3.4 (decode the deterministic sections once, then fork), and the bounded wait of the
attention kernel's merge."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import MASKED
from oracle.cache import ForkSet
from oracle.jmt import average_rollouts_jmt
from oracle.unmask import unmask_step
from paper_2605_23163_b200 import fdd, harness, synth

import parity_utils as pu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _need_cuda():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    fdd.lib()


def _attn(ctx, forkset, layer, q, k, v, d, causal=False, head_dim=128):
    qd, kd, vd = harness.bf16_tensor(q), harness.bf16_tensor(k), harness.bf16_tensor(v)
    out = torch.full_like(qd, float("nan"))
    fdd.fdd_block_attn(ctx, [forkset], layer, qd, kd, vd, out, [d], 1.0 / np.sqrt(head_dim), int(causal))
    fdd.fdd_poll_status(ctx)
    return out.float().cpu().numpy().astype(np.float64)


def _oracle_attn(w, ofs, layer, q, k, v):
    return pu.attention_oracle(w, (ofs.prefix_k[layer], ofs.prefix_v[layer]),
                               (ofs.suffix_k[layer], ofs.suffix_v[layer]), q, k, v)


def test_three_layers_with_caches_of_their_own():
    # Sec. 3.3: the caches of earlier blocks are reused, layer by layer.  Three layers with distinct
    # prefix and suffix caches; two blocks; attention on every layer against that layer's oracle
    # cache; the suffix length advances only with the last layer's commit; a second fork over the
    # same buffers (the tensor maps of the freed set serve again) reads the same caches.
    L = 3
    w = synth.small_variant(synth.workload("tts"), prefix_len=700 + 29, vocab=512, n_forks=3, n_blocks=3)
    sc = w.scenes[0]
    d = sc.block_len
    ctx = harness.create_context(w, n_layers=L)
    try:
        scene = harness.GpuScene(ctx, w, 0, n_layers=L, suffix_capacity=3 * d)
        prefixes = [synth.make_prefix(w, 0, layer) for layer in range(L)]
        assert not np.array_equal(prefixes[0][0], prefixes[1][0])
        ofs = ForkSet([p[0] for p in prefixes], [p[1] for p in prefixes], sc.n_forks, scene.seeds)
        for block in range(2):
            per_layer = [synth.make_qkv(w, 0, layer, block, 0) for layer in range(L)]
            for layer in (2, 0, 1):                        # any order: a layer reads its own caches only
                q, k, v = per_layer[layer]
                got = _attn(ctx, scene.forkset, layer, q, k, v, d)
                pu.assert_attention_close(got, _oracle_attn(w, ofs, layer, q, k, v))
            for layer in range(L):
                _, k, v = per_layer[layer]
                fdd.fdd_kv_commit(ctx, [scene.forkset], layer, harness.bf16_tensor(k), harness.bf16_tensor(v), [d],
                                  1 if layer == L - 1 else 0)
                # every layer of a block is written at the same place: the length moves with the last one
                assert fdd.fdd_forkset_suffix_len(scene.forkset) == ((block + 1) * d if layer == L - 1 else block * d)
                ofs.kv_commit(layer, k, v)
        fdd.fdd_poll_status(ctx)
        for layer in range(L):                             # the bytes landed in the right layer's buffer
            sk = scene.suffix_k[layer].view(torch.int16).cpu().numpy().view(np.uint16)
            for f in range(sc.n_forks):
                assert np.array_equal(sk[f, :, :2 * d].transpose(1, 0, 2), ofs.suffix_k[layer][f])
        # free, fork again over the same buffers, put the two blocks back, and read every layer
        scene.free()
        again = fdd.fdd_fork(ctx, scene.prefix_k, scene.prefix_v, None, sc.prefix_len, scene.prefix_capacity,
                             sc.n_forks, scene.seeds, scene.suffix_k, scene.suffix_v, scene.suffix_capacity)
        assert fdd.fdd_forkset_suffix_len(again) == 0
        for block in range(2):
            for layer in range(L):
                _, k, v = synth.make_qkv(w, 0, layer, block, 0)
                fdd.fdd_kv_commit(ctx, [again], layer, harness.bf16_tensor(k), harness.bf16_tensor(v), [d],
                                  1 if layer == L - 1 else 0)
        for layer in range(L):
            q, k, v = synth.make_qkv(w, 0, layer, 2, 1)
            got = _attn(ctx, again, layer, q, k, v, d)
            pu.assert_attention_close(got, _oracle_attn(w, ofs, layer, q, k, v))
        with pytest.raises(fdd.FddError) as ei:
            fdd.fdd_block_attn(ctx, [again], L, harness.bf16_tensor(q), harness.bf16_tensor(k), harness.bf16_tensor(v),
                               torch.empty_like(harness.bf16_tensor(q)), [d], 0.1, 0)
        assert ei.value.status == fdd.FDD_ERR_SHAPE
    finally:
        fdd.fdd_destroy(ctx)


def _decode_block_both(ctx, w, forkset, ofs, block, n, seeds, temperature, sample=None):
    """One block loop on the GPU and in the oracle, step by step from the oracle's state; returns
    the final tokens / state and the last step's K/V."""
    sc = w.scenes[0]
    tokens, state = synth.make_block_template(w, 0, block)
    tokens, state = tokens[:n].copy(), state[:n].copy()
    step, ambiguous = 0, 0
    k = v = None
    while np.any(state == MASKED):
        q, k, v = (x[:n] for x in synth.make_qkv(w, 0, 0, block, step))
        got_attn = _attn(ctx, forkset, 0, q, k, v, sc.block_len)
        pu.assert_attention_close(got_attn, _oracle_attn(w, ofs, 0, q, k, v))
        logits = synth.make_logits(w, 0, block, step, rows="all")[:n]
        tok_d = torch.from_numpy(tokens).cuda()
        st_d = torch.from_numpy(state).cuda()
        n_c = torch.zeros(n, dtype=torch.int32, device="cuda")
        n_l = torch.zeros(n, dtype=torch.int32, device="cuda")
        conf = torch.zeros(tokens.shape, dtype=torch.float32, device="cuda")
        fdd.fdd_unmask(ctx, [forkset], harness.logits_tensor(w, logits), tok_d, st_d, [sc.block_len], w.threshold,
                       temperature, block, step, n_c, n_l, conf)
        fdd.fdd_poll_status(ctx)
        got = dict(tokens=tok_d.cpu().numpy(), state=st_d.cpu().numpy(), n_committed=n_c.cpu().numpy(),
                   n_left=n_l.cpu().numpy(), conf=conf.cpu().numpy())
        ref = unmask_step(pu.widen_logits(w, logits), tokens, state, seeds, w.threshold, temperature, block, step)
        ambiguous += len(pu.compare_unmask(got, ref, tokens, state, w.threshold)["ambiguous_forks"])
        tokens, state = ref["tokens"], ref["state"]
        step += 1
        assert step <= sc.block_len
    assert ambiguous <= 2
    return tokens, state, k, v


@pytest.mark.parametrize("paged", [False, True])
def test_scene_decodes_deterministic_blocks_once_then_forks(paged):
    # Sec. 3.4: three greedy blocks by one rollout, each committed to the shared prefix itself; then
    # eight rollouts forked from that cache (nothing copied) decode three sampled blocks with private
    # suffixes; their trajectories are interpolated and averaged.  Every attention and unmasking step
    # is held against the oracle, which does the same thing on arrays.
    base = synth.workload("tts")
    P = 64 * 9 + 17 if paged else 4096
    sc = synth.Scene(prefix_len=P, n_forks=8, block_len=32, n_scaffold=10, n_blocks=6)
    w = synth.Workload("scene", base.n_q_heads, base.n_kv_heads, base.head_dim, 2048 * 5 + 1024, "bf16", "peaked",
                       0.9, 1.0, (sc,), page_tokens=64 if paged else 0, seed=41)
    d, N = sc.block_len, sc.n_forks
    ctx = harness.create_context(w)
    try:
        pk, pv = synth.make_prefix(w, 0)
        cap_tokens = P + 3 * d
        if paged:
            n_pages = (cap_tokens + 63) // 64
            pool = n_pages + 2
            ids = synth.page_order(w, 0, n_pages, pool)
            table = torch.from_numpy(ids).cuda()
            dk = harness.pack_prefix_paged(pk, 64, ids, pool)
            dv = harness.pack_prefix_paged(pv, 64, ids, pool)
            capacity = pool
        else:
            table = None
            dk = harness.pack_prefix_contiguous(pk, cap_tokens)
            dv = harness.pack_prefix_contiguous(pv, cap_tokens)
            capacity = cap_tokens
        seeds = synth.fork_seeds(w, 0)
        shape1 = (1, w.n_kv_heads, d, w.head_dim)
        s1k, s1v = (torch.zeros(shape1, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        one = fdd.fdd_fork(ctx, [dk], [dv], table, P, capacity, 1, seeds[:1], [s1k], [s1v], d)
        o_one = ForkSet([pk], [pv], 1, seeds[:1])
        finished = []
        for block in range(3):                             # the deterministic sections: greedy, one rollout
            tokens, state, k, v = _decode_block_both(ctx, w, one, o_one, block, 1, seeds[:1], 0.0)
            finished.append((tokens, state))
            fdd.fdd_prefix_extend(ctx, [one], 0, harness.bf16_tensor(k), harness.bf16_tensor(v), [d], 1)
            o_one.extend_prefix(0, k, v)
            assert fdd.fdd_forkset_prefix_len(one) == P + (block + 1) * d
        fdd.fdd_poll_status(ctx)
        assert fdd.fdd_forkset_suffix_len(one) == 0
        if not paged:                                      # the contiguous cache is full now (the page pool has spare pages)
            with pytest.raises(fdd.FddError) as ei:
                fdd.fdd_prefix_extend(ctx, [one], 0, harness.bf16_tensor(k), harness.bf16_tensor(v), [d], 1)
            assert ei.value.status == fdd.FDD_ERR_CAPACITY
        P2 = fdd.fdd_forkset_prefix_len(one)
        # fork: same cache buffers, longer prefix
        shapeN = (N, w.n_kv_heads, 3 * d, w.head_dim)
        sNk, sNv = (torch.zeros(shapeN, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        many = fdd.fdd_fork(ctx, [dk], [dv], table, P2, capacity, N, seeds, [sNk], [sNv], 3 * d)
        o_many = o_one.fork(N, seeds)
        with pytest.raises(fdd.FddError) as ei:            # only a set of one rollout extends the prefix
            fdd.fdd_prefix_extend(ctx, [many], 0, harness.bf16_tensor(k), harness.bf16_tensor(v), [d], 1)
        assert ei.value.status == fdd.FDD_ERR_STATE
        traj_tokens, traj_state = [], []
        for block in range(3, 6):                          # the trajectory section: sampled, N rollouts
            tokens, state, k, v = _decode_block_both(ctx, w, many, o_many, block, N, seeds, w.temperature)
            traj_tokens.append(tokens)
            traj_state.append(state)
            fdd.fdd_kv_commit(ctx, [many], 0, harness.bf16_tensor(k), harness.bf16_tensor(v), [d], 1)
            o_many.kv_commit(0, k, v)
        assert fdd.fdd_forkset_suffix_len(many) == 3 * d
        # rollouts differ (independent draws) although they share every cached token before the fork
        assert len({tuple(t.tolist()) for t in np.concatenate(traj_tokens, axis=1)}) > 1
        traj = synth.tokens_to_trajectory(w, np.concatenate(traj_tokens, axis=1), np.concatenate(traj_state, axis=1))
        out = torch.zeros((20, 2), dtype=torch.float32, device="cuda")
        fdd.fdd_average_rollouts_jmt(ctx, torch.from_numpy(traj).cuda(), N, w.waypoints, 20, out)
        fdd.fdd_poll_status(ctx)
        ref = average_rollouts_jmt(traj, 20)
        assert np.allclose(out.cpu().numpy(), ref, rtol=1e-5, atol=1e-5 * np.abs(ref).max())
    finally:
        fdd.fdd_destroy(ctx)


def test_merge_wait_that_runs_out_is_reported_and_the_context_recovers():
    # One rollout, one KV head, head dimension 64 over a 10000-token prefix: a single unit of work cut
    # into about ten pieces, whose holders wait for one another before they merge.  With a wait limit
    # of one clock the first CTA to finish gives up at once: the launch still ends, the status word
    # says FDD_ERR_DEVICE_TIMEOUT, reading it puts the counters back in order, and the next call on
    # the same context matches the oracle.  (Its limit is long, but not the default one: then the unit would go to a cluster,
    # whose merge has no counters.)
    sc = synth.Scene(prefix_len=10000, n_forks=1, block_len=16, n_scaffold=4, n_blocks=1)
    w = synth.Workload("d64_wait", 4, 1, 64, 256, "f32", "normal_sigma2", 0.9, 0.0, (sc,), qkv_sigma=0.35, seed=77)
    ctx = harness.create_context(w)
    try:
        scene = harness.GpuScene(ctx, w, 0)
        pk, pv = synth.make_prefix(w, 0)
        ofs = ForkSet([pk], [pv], 1, scene.seeds)
        q, k, v = synth.make_qkv(w, 0, 0, 0, 0)
        fdd.fdd_set_merge_wait_limit(ctx, 1)
        qd, kd, vd = harness.bf16_tensor(q), harness.bf16_tensor(k), harness.bf16_tensor(v)
        out = torch.full_like(qd, float("nan"))
        fdd.fdd_block_attn(ctx, [scene.forkset], 0, qd, kd, vd, out, [sc.block_len], 0.125, 0)
        with pytest.raises(fdd.FddError) as ei:
            fdd.fdd_poll_status(ctx)
        assert ei.value.status == fdd.FDD_ERR_DEVICE_TIMEOUT
        fdd.fdd_poll_status(ctx)                           # read and cleared
        with pytest.raises(fdd.FddError):
            fdd.fdd_set_merge_wait_limit(ctx, 0)
        fdd.fdd_set_merge_wait_limit(ctx, 3_999_999_999)
        for _ in range(2):
            got = _attn(ctx, scene.forkset, 0, q, k, v, sc.block_len, head_dim=64)
            pu.assert_attention_close(got, _oracle_attn(w, ofs, 0, q, k, v))
    finally:
        fdd.fdd_destroy(ctx)


def test_library_block_loop_matches_the_oracle_loop():
    # Sec. 3.3: fdd_decode_block runs the denoising loop of a block by itself (gated attention on
    # every layer, unmasking, counts to the host, one step ahead) and commits the block's K/V when no
    # MASK is left.  Two layers with caches of their own, two blocks in a row (the second reads what
    # the first committed).  The oracle runs its own loop on the same inputs: the number of steps,
    # the final tokens and state, the attention output of every step for the rollouts that still
    # decoded, and the committed bytes must agree; rollouts that had finished are never written.
    from oracle.decode import decode_block
    L = 2
    w = synth.small_variant(synth.workload("tts"), prefix_len=300 + 11, vocab=2048, n_forks=5, n_blocks=2)
    sc = w.scenes[0]
    N, d = sc.n_forks, sc.block_len
    scale = 1.0 / np.sqrt(w.head_dim)
    ctx = harness.create_context(w, n_layers=L)
    try:
        scene = harness.GpuScene(ctx, w, 0, n_layers=L, suffix_capacity=2 * d)
        prefixes = [synth.make_prefix(w, 0, layer) for layer in range(L)]
        ofs = ForkSet([p[0] for p in prefixes], [p[1] for p in prefixes], N, scene.seeds)
        for block in range(2):
            tokens0, state0 = synth.make_block_template(w, 0, block)
            steps_in = d                                   # a block never needs more steps than it has positions
            host = [dict(qkv=[synth.make_qkv(w, 0, layer, block, t) for layer in range(L)],
                         logits=synth.make_logits(w, 0, block, t, rows="all")) for t in range(steps_in)]
            inputs = lambda t: dict(q=[x[0] for x in host[t]["qkv"]], k=[x[1] for x in host[t]["qkv"]],
                                    v=[x[2] for x in host[t]["qkv"]], logits=host[t]["logits"])
            ref = decode_block(ofs, inputs, tokens0, state0, w.threshold, w.temperature, block, scale)
            dq = [[harness.bf16_tensor(x[0]) for x in h["qkv"]] for h in host]
            dk = [[harness.bf16_tensor(x[1]) for x in h["qkv"]] for h in host]
            dv = [[harness.bf16_tensor(x[2]) for x in h["qkv"]] for h in host]
            dout = [[torch.full_like(q_, float("nan")) for q_ in per] for per in dq]
            dlg = [harness.logits_tensor(w, h["logits"]) for h in host]
            tokens = torch.from_numpy(tokens0).cuda()
            state = torch.from_numpy(state0).cuda()
            n_c = torch.zeros(N, dtype=torch.int32, device="cuda")
            n_l = torch.zeros(N, dtype=torch.int32, device="cuda")
            steps, left = fdd.fdd_decode_block(ctx, [scene.forkset], L, steps_in, dq, dk, dv, dout, dlg, tokens, state,
                                               [d], scale, 0, w.threshold, w.temperature, block, 1, n_c, n_l)
            fdd.fdd_poll_status(ctx)
            assert left == 0 and steps == ref["steps"] and 2 <= steps < d
            assert np.array_equal(state.cpu().numpy(), ref["state"]) and not np.any(ref["state"] == MASKED)
            assert np.array_equal(tokens.cpu().numpy(), ref["tokens"])
            assert fdd.fdd_forkset_suffix_len(scene.forkset) == (block + 1) * d
            # attention of every step: who still decoded on entry follows from the oracle's commits
            masked_left = (state0 == MASKED).sum(axis=1)
            for t in range(steps + 1):                     # the step after the last one was issued ahead and must do nothing
                decoding = np.nonzero(masked_left > 0)[0] if t < steps else np.zeros(0, dtype=int)
                for layer in range(L):
                    got = dout[t][layer].float().cpu().numpy().astype(np.float64).reshape(N, d, w.n_q_heads, w.head_dim)
                    if t < steps:
                        pu.assert_attention_close(got[decoding], ref["attn"][t][layer][decoding])
                    idle = np.setdiff1d(np.arange(N), decoding)
                    assert np.all(np.isnan(got[idle])), "attention wrote rows of a rollout that had finished"
                if t < steps:
                    masked_left = masked_left - ref["committed_per_step"][t]
            for layer in range(L):                         # the committed bytes (the oracle's loop commits too)
                sk = scene.suffix_k[layer].view(torch.int16).cpu().numpy().view(np.uint16)
                for f in range(N):
                    assert np.array_equal(sk[f, :, :(block + 1) * d].transpose(1, 0, 2), ofs.suffix_k[layer][f])
        # a loop that is cut short says so and commits nothing
        tokens0, state0 = synth.make_block_template(w, 0, 0)
        tokens, state = torch.from_numpy(tokens0).cuda(), torch.from_numpy(state0).cuda()
        before = fdd.fdd_forkset_suffix_len(scene.forkset)
        steps, left = fdd.fdd_decode_block(ctx, [scene.forkset], L, 1, dq[:1], dk[:1], dv[:1], dout[:1], dlg[:1], tokens, state,
                                           [d], scale, 0, w.threshold, w.temperature, 0, 1, n_c, n_l)
        fdd.fdd_poll_status(ctx)
        assert steps == 1 and left == int((state.cpu().numpy() == MASKED).sum()) > 0
        assert fdd.fdd_forkset_suffix_len(scene.forkset) == before
        # argument errors come back before anything is issued
        launches = fdd.fdd_launch_count(ctx)
        for bad in (dict(n_layers=L + 1), dict(max_steps=0)):
            with pytest.raises(fdd.FddError) as ei:
                fdd.fdd_decode_block(ctx, [scene.forkset], bad.get("n_layers", L), bad.get("max_steps", 1), dq[:1], dk[:1], dv[:1],
                                     dout[:1], dlg[:1], tokens, state, [d], scale, 0, w.threshold, w.temperature, 0, 1, n_c, n_l)
            assert ei.value.status == fdd.FDD_ERR_INVALID_ARG
        assert fdd.fdd_launch_count(ctx) == launches
    finally:
        fdd.fdd_destroy(ctx)


def test_library_block_loop_with_more_scenes_than_one_unmask_launch_takes():
    # Eighteen small scenes (different rollouts, block lengths and prefix lengths) in one
    # fdd_decode_block call: the unmasking step splits them into two launches, whose counts must all
    # reach the loop's host buffer at the right place.  Every scene against the oracle's own loop.
    from oracle.decode import decode_block
    base = synth.workload("serving_mix")
    rng = np.random.default_rng(7)
    scenes = tuple(synth.Scene(int(rng.integers(1, 200)), int(rng.integers(1, 4)), int(rng.choice([16, 32])),
                               int(rng.integers(3, 9)), 1) for _ in range(18))
    w = synth.Workload("mix_loop", base.n_q_heads, base.n_kv_heads, base.head_dim, 512, "bf16", "peaked", 0.9, 1.0,
                       scenes, page_tokens=64, seed=23)
    scale = 1.0 / np.sqrt(w.head_dim)
    d_max = max(sc.block_len for sc in scenes)
    ctx = harness.create_context(w)
    try:
        gs = [harness.GpuScene(ctx, w, i, suffix_capacity=sc.block_len) for i, sc in enumerate(scenes)]
        refs, host_steps = [], [[] for _ in range(d_max)]
        tokens0, state0 = [], []
        for i, sc in enumerate(scenes):
            pk, pv = synth.make_prefix(w, i)
            ofs = ForkSet([pk], [pv], sc.n_forks, gs[i].seeds)
            t0, s0 = synth.make_block_template(w, i, 0)
            per_step = [dict(qkv=synth.make_qkv(w, i, 0, 0, t), logits=synth.make_logits(w, i, 0, t, rows="all"))
                        for t in range(d_max)]
            inputs = lambda t, ps=per_step: dict(q=[ps[t]["qkv"][0]], k=[ps[t]["qkv"][1]], v=[ps[t]["qkv"][2]],
                                                 logits=ps[t]["logits"])
            refs.append(decode_block(ofs, inputs, t0, s0, w.threshold, w.temperature, 0, scale, want_attention=False))
            for t in range(d_max):
                host_steps[t].append(per_step[t])
            tokens0.append(t0.reshape(-1)); state0.append(s0.reshape(-1))
        pack = lambda xs: np.concatenate([np.asarray(x).reshape(-1) for x in xs])
        dq = [[harness.bf16_tensor(pack([p["qkv"][0] for p in host_steps[t]]))] for t in range(d_max)]
        dk = [[harness.bf16_tensor(pack([p["qkv"][1] for p in host_steps[t]]))] for t in range(d_max)]
        dv = [[harness.bf16_tensor(pack([p["qkv"][2] for p in host_steps[t]]))] for t in range(d_max)]
        dout = [[torch.empty_like(x[0])] for x in dq]
        dlg = [harness.logits_tensor(w, pack([p["logits"] for p in host_steps[t]])) for t in range(d_max)]
        tokens = torch.from_numpy(np.concatenate(tokens0)).cuda()
        state = torch.from_numpy(np.concatenate(state0)).cuda()
        N = sum(sc.n_forks for sc in scenes)
        n_c = torch.zeros(N, dtype=torch.int32, device="cuda")
        n_l = torch.zeros(N, dtype=torch.int32, device="cuda")
        steps, left = fdd.fdd_decode_block(ctx, [g.forkset for g in gs], 1, d_max, dq, dk, dv, dout, dlg, tokens, state,
                                           [sc.block_len for sc in scenes], scale, 0, w.threshold, w.temperature, 0, 1,
                                           n_c, n_l)
        fdd.fdd_poll_status(ctx)
        assert left == 0 and steps == max(r["steps"] for r in refs)
        got_tok, got_st = tokens.cpu().numpy(), state.cpu().numpy()
        off = 0
        for sc, ref, g in zip(scenes, refs, gs):
            n = sc.n_forks * sc.block_len
            assert np.array_equal(got_st[off:off + n].reshape(ref["state"].shape), ref["state"])
            assert np.array_equal(got_tok[off:off + n].reshape(ref["tokens"].shape), ref["tokens"])
            assert fdd.fdd_forkset_suffix_len(g.forkset) == sc.block_len
            off += n
    finally:
        fdd.fdd_destroy(ctx)


@pytest.mark.parametrize("layers,shared", [(2, ""), (18, ""), (50, ""), (3, "one output"), (3, "output feeds the next layer"),
                                           (3, "one suffix cache")])
def test_library_block_loop_does_what_calls_layer_by_layer_do(layers, shared):
    # The layers of a step go to the GPU together where none touches what another writes, one behind the other
    # elsewhere; either way the result is that of the calls made one by one.  50 layers take four attention launches
    # and two appends.
    hq, hkv, dim, vocab, n, d, prefix = 8, 2, 64, 512, 3, 16, 300
    scale = 1.0 / np.sqrt(dim)

    def decode(by_library):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(5)
        normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
        ctx = fdd.fdd_create(hq, hkv, dim, vocab, layers, 0, d, n, fdd.FDD_LOGITS_BF16)
        try:
            pk, pv = normal(layers, hkv, prefix, dim), normal(layers, hkv, prefix, dim)
            sk, sv = (torch.zeros((layers, n, hkv, 2 * d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
            q, out = [normal(n * d * hq * dim) for _ in range(layers)], [torch.full((n * d * hq * dim,), float("nan"), dtype=torch.bfloat16, device="cuda")
                                                                         for _ in range(layers)]
            k, v = [normal(n * d * hkv * dim) for _ in range(layers)], [normal(n * d * hkv * dim) for _ in range(layers)]
            logits = 2.0 * torch.randn((n * d, vocab), generator=gen, device="cuda").to(torch.bfloat16)
            suffix_k = [sk[0]] * layers if shared == "one suffix cache" else list(sk)
            if shared == "one output":
                out = [out[0]] * layers
            elif shared == "output feeds the next layer":
                out = q[1:] + out[-1:]
            forkset = fdd.fdd_fork(ctx, list(pk), list(pv), None, prefix, prefix, n, [11, 12, 13], suffix_k, list(sv), 2 * d)
            for block in range(2):
                tokens = torch.full((n * d,), vocab - 1, dtype=torch.int32, device="cuda")
                state = torch.full((n * d,), MASKED, dtype=torch.uint8, device="cuda")
                state.view(n, d)[1, 4:] = fdd.FDD_COMMITTED          # this rollout is through long before the others
                n_c, n_l = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
                if by_library:
                    fdd.fdd_decode_block(ctx, [forkset], layers, d, [q], [k], [v], [out], [logits], tokens, state, [d], scale, 0, 0.9, 0.0,
                                         block, 1, n_c, n_l)
                    continue
                for t in range(d):
                    for layer in range(layers):
                        fdd.fdd_block_attn_gated(ctx, [forkset], layer, q[layer], k[layer], v[layer], out[layer], [d], scale, 0,
                                                 n_l if t else None)
                    fdd.fdd_unmask(ctx, [forkset], logits, tokens, state, [d], 0.9, 0.0, block, t, n_c, n_l, None)
                    if int(n_l.sum()) == 0:
                        break
                for layer in range(layers):
                    fdd.fdd_kv_commit(ctx, [forkset], layer, k[layer], v[layer], [d], 1 if layer == layers - 1 else 0)
            fdd.fdd_poll_status(ctx)
            return torch.stack(out).float().cpu().numpy().astype(np.float64), tokens.cpu(), state.cpu(), sk.cpu(), sv.cpu()
        finally:
            fdd.fdd_destroy(ctx)

    got, ref = decode(True), decode(False)
    pu.assert_attention_close(got[0], ref[0])
    for a, b in zip(got[1:], ref[1:]):
        assert torch.equal(a, b)


def test_library_block_loop_leaves_the_stream_behind_its_attention():
    # The attention may run on a stream of its own: what the caller enqueues after the call still comes behind it, and
    # what the call refuses it refuses before anything of the step has happened.
    hq, hkv, dim, vocab, n, d, prefix = 16, 2, 128, 512, 4, 32, 4000
    scale = 1.0 / np.sqrt(dim)
    ctx = fdd.fdd_create(hq, hkv, dim, vocab, 1, 0, d, n, fdd.FDD_LOGITS_BF16)
    try:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            gen = torch.Generator(device="cuda")
            gen.manual_seed(6)
            normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
            pk, pv = normal(hkv, prefix, dim), normal(hkv, prefix, dim)
            sk, sv = (torch.zeros((n, hkv, d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
            forkset = fdd.fdd_fork(ctx, [pk], [pv], None, prefix, prefix, n, [1, 2, 3, 4], [sk], [sv], d)
            q, k, v = normal(n * d * hq * dim), normal(n * d * hkv * dim), normal(n * d * hkv * dim)
            logits = 2.0 * normal(n * d, vocab)
            ref = torch.zeros_like(q)
            fdd.fdd_block_attn(ctx, [forkset], 0, q, k, v, ref, [d], scale, 0)
            tokens = torch.full((n * d,), -1, dtype=torch.int32, device="cuda")
            state = torch.full((n * d,), MASKED, dtype=torch.uint8, device="cuda")
            n_c, n_l = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
            odd = torch.zeros(q.numel() + 1, dtype=torch.bfloat16, device="cuda")[1:]
            launches = fdd.fdd_launch_count(ctx)
            for bad in (dict(q=odd), dict(out=odd), dict(scale=0.0)):
                with pytest.raises(fdd.FddError) as ei:
                    fdd.fdd_decode_block(ctx, [forkset], 1, d, [[bad.get("q", q)]], [[k]], [[v]], [[bad.get("out", ref)]], [logits], tokens,
                                         state, [d], bad.get("scale", scale), 0, 0.9, 0.0, 0, 0, n_c, n_l)
                assert ei.value.status == fdd.FDD_ERR_INVALID_ARG
            assert fdd.fdd_launch_count(ctx) == launches and bool((state == MASKED).all())
            for _ in range(10):
                qq, out = q.clone(), torch.zeros_like(q)
                state.fill_(MASKED)
                fdd.fdd_decode_block(ctx, [forkset], 1, d, [[qq]], [[k]], [[v]], [[out]], [logits], tokens, state, [d], scale, 0, 0.9, 0.0,
                                     0, 0, n_c, n_l)
                got = out.clone()                          # behind the last step's attention
                qq.zero_()                                 # and so is this
                out.zero_()
                stream.synchronize()
                assert bool((got != 0).any(dim=0).any())
                pu.assert_attention_close(got.float().cpu().numpy().astype(np.float64), ref.float().cpu().numpy().astype(np.float64))
                assert not bool(out.any())
        fdd.fdd_poll_status(ctx)
    finally:
        fdd.fdd_destroy(ctx)


def _attention64(q, k, v, pk, pv, scale):
    """Attention of one layer in 64 bits: q [n, d, hq, dim], k and v [n, d, hkv, dim], pk and pv [hkv, prefix, dim]."""
    n, d, hq, dim = q.shape
    hkv = k.shape[2]
    res = []
    for f in range(n):
        keys, vals = (torch.cat([p.double(), x[f].double().transpose(0, 1)], 1) for p, x in ((pk, k), (pv, v)))
        qh = q[f].double().view(d, hkv, hq // hkv, dim).permute(1, 2, 0, 3).reshape(hkv, -1, dim)
        o = torch.softmax(qh @ keys.transpose(1, 2) * scale, -1) @ vals
        res.append(o.view(hkv, hq // hkv, d, dim).permute(2, 0, 1, 3).reshape(d, hq, dim))
    return torch.stack(res)


@pytest.mark.parametrize("layers,forks,prefix", [
    (1, 1, 4096),        # a piece per tile step -> clusters of sixteen
    (1, 8, 4096),        # pieces of four tile steps -> clusters of four
    (1, 20, 2500),       # pieces of six -> of eleven, beside the unmasking
    (6, 8, 4003),        # pieces of four -> layers together, up to whole units
    (6, 1, 1500),
])
def test_longer_pieces_are_as_precise_as_the_finer_cut(layers, forks, prefix):
    # The error against 64 bits goes with how often a row's reference is the maximum of the tile at hand; launches that
    # cut longer pieces than a layer by itself on all SMs take the reference anew.  The finer cut is what a call takes that has a wait
    # limit of its own.  The two errors are of the same distribution then, over 65536 values or more a layer: 1 % is four
    # times their scatter, and half of what is lost (2.7 to 4.5 %) if a piece keeps its first reference.
    hq, hkv, dim, d, vocab = 16, 2, 128, 32, 512
    scale = 1.0 / np.sqrt(dim)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(prefix + forks)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
    pk, pv = normal(layers, hkv, prefix, dim), normal(layers, hkv, prefix, dim)
    sk, sv = (torch.zeros((layers, forks, hkv, d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    q, k, v = normal(layers, forks, d, hq, dim), normal(layers, forks, d, hkv, dim), normal(layers, forks, d, hkv, dim)
    exact = torch.stack([_attention64(q[l], k[l], v[l], pk[l], pv[l], scale) for l in range(layers)])
    error = lambda out: float(torch.linalg.vector_norm(out.double() - exact) / torch.linalg.vector_norm(exact))
    ctx = fdd.fdd_create(hq, hkv, dim, vocab, layers, 0, d, forks, fdd.FDD_LOGITS_BF16)
    try:
        forkset = fdd.fdd_fork(ctx, list(pk), list(pv), None, prefix, prefix, forks, list(range(forks)), list(sk), list(sv), d)
        finer, called, looped = (torch.full_like(q, float("nan")) for _ in range(3))
        fdd.fdd_set_merge_wait_limit(ctx, 3_999_999_999)
        for l in range(layers):
            fdd.fdd_block_attn(ctx, [forkset], l, q[l], k[l], v[l], finer[l], [d], scale, 0)
        fdd.fdd_set_merge_wait_limit(ctx, 4_000_000_000)
        for l in range(layers):
            fdd.fdd_block_attn(ctx, [forkset], l, q[l], k[l], v[l], called[l], [d], scale, 0)
        tokens = torch.zeros(forks * d, dtype=torch.int32, device="cuda")
        state = torch.full((forks * d,), MASKED, dtype=torch.uint8, device="cuda")
        n_c, n_l = (torch.zeros(forks, dtype=torch.int32, device="cuda") for _ in range(2))
        fdd.fdd_decode_block(ctx, [forkset], layers, 1, [list(q)], [list(k)], [list(v)], [list(looped)], [normal(forks * d, vocab)], tokens,
                             state, [d], scale, 0, 0.9, 0.0, 0, 0, n_c, n_l)
        fdd.fdd_poll_status(ctx)
        for out in (called, looped):
            assert error(out) <= 1.01 * error(finer), (error(out), error(finer))
    finally:
        fdd.fdd_destroy(ctx)


def test_context_for_many_rollouts_and_layers():
    # 24 layers times 128 units of each of 700,000 rollouts are more than 2^31 counters: a context keeps no more than one
    # layer takes, and launches hold as many layers as that leaves room for.
    hq, hkv, dim, d, layers, n, prefix = 128, 8, 64, 128, 24, 1, 130
    ctx = fdd.fdd_create(hq, hkv, dim, 512, layers, 0, d, 700_000, fdd.FDD_LOGITS_BF16)
    try:
        gen = torch.Generator(device="cuda")
        gen.manual_seed(7)
        normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
        pk, pv = normal(layers, hkv, prefix, dim), normal(layers, hkv, prefix, dim)
        sk, sv = (torch.zeros((layers, n, hkv, d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        q, k, v = normal(layers, n, d, hq, dim), normal(layers, n, d, hkv, dim), normal(layers, n, d, hkv, dim)
        out = torch.full_like(q, float("nan"))
        forkset = fdd.fdd_fork(ctx, list(pk), list(pv), None, prefix, prefix, n, [1], list(sk), list(sv), d)
        tokens, state = torch.zeros(d, dtype=torch.int32, device="cuda"), torch.full((d,), MASKED, dtype=torch.uint8, device="cuda")
        n_c, n_l = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
        fdd.fdd_decode_block(ctx, [forkset], layers, 2, [list(q)], [list(k)], [list(v)], [list(out)], [normal(d, 512)], tokens, state, [d],
                             dim ** -0.5, 0, 0.9, 0.0, 0, 0, n_c, n_l)
        fdd.fdd_poll_status(ctx)
        for l in (0, layers - 1):
            ref = _attention64(q[l], k[l], v[l], pk[l], pv[l], dim ** -0.5)
            pu.assert_attention_close(out[l].float().cpu().numpy().astype(np.float64), ref.cpu().numpy())
    finally:
        fdd.fdd_destroy(ctx)


def test_library_block_loop_on_streams_of_any_priority():
    # The stream that the attention runs on has the priority of the caller's; several of them may be in use in turn.
    hq, hkv, dim, vocab, n, d, prefix = 16, 2, 128, 512, 4, 16, 1000
    ctx = fdd.fdd_create(hq, hkv, dim, vocab, 1, 0, d, n, fdd.FDD_LOGITS_BF16)
    try:
        gen = torch.Generator(device="cuda")
        gen.manual_seed(8)
        normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
        pk, pv = normal(hkv, prefix, dim), normal(hkv, prefix, dim)
        sk, sv = (torch.zeros((n, hkv, d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        forkset = fdd.fdd_fork(ctx, [pk], [pv], None, prefix, prefix, n, [1, 2, 3, 4], [sk], [sv], d)
        q, k, v, logits = normal(n, d, hq, dim), normal(n, d, hkv, dim), normal(n, d, hkv, dim), normal(n * d, vocab)
        ref = _attention64(q, k, v, pk, pv, dim ** -0.5).cpu().numpy()
        torch.cuda.synchronize()
        seen = []
        for priority in (0, -1, -3, 0, -1):
            stream = torch.cuda.Stream(priority=priority)
            with torch.cuda.stream(stream):
                out = torch.full_like(q, float("nan"))
                tokens = torch.zeros(n * d, dtype=torch.int32, device="cuda")
                state = torch.full((n * d,), MASKED, dtype=torch.uint8, device="cuda")
                n_c, n_l = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
                steps, left = fdd.fdd_decode_block(ctx, [forkset], 1, d, [[q]], [[k]], [[v]], [[out]], [logits], tokens, state, [d], dim ** -0.5,
                                                   0, 0.9, 0.0, 0, 0, n_c, n_l)
                got = out.float().cpu().numpy().astype(np.float64)
            assert left == 0
            pu.assert_attention_close(got, ref)
            seen.append((steps, tokens.cpu().tolist()))
        assert all(x == seen[0] for x in seen)
        fdd.fdd_poll_status(ctx)
    finally:
        fdd.fdd_destroy(ctx)


def test_library_block_loop_with_a_callback_that_makes_each_steps_inputs():
    # A model in the loop writes every step into the same buffers, from the callback.  The result is that of the loop
    # which finds each step's inputs in buffers of their own.
    hq, hkv, dim, vocab, layers, n, d, prefix = 16, 2, 128, 1024, 2, 3, 24, 700
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
    pk, pv = normal(layers, hkv, prefix, dim), normal(layers, hkv, prefix, dim)
    Q, K, V = normal(d, layers, n, d, hq, dim), normal(d, layers, n, d, hkv, dim), normal(d, layers, n, d, hkv, dim)
    S = 3.0 * normal(d, n * d, vocab)
    S[:, torch.arange(n * d), torch.arange(n * d)] += 12.0 * torch.rand((d, n * d), generator=gen, device="cuda")

    def decode(callback):
        ctx = fdd.fdd_create(hq, hkv, dim, vocab, layers, 0, d, n, fdd.FDD_LOGITS_BF16)
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                sk, sv = (torch.zeros((layers, n, hkv, d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
                forkset = fdd.fdd_fork(ctx, list(pk), list(pv), None, prefix, prefix, n, [5, 6, 7], list(sk), list(sv), d)
                tokens = torch.zeros(n * d, dtype=torch.int32, device="cuda")
                state = torch.full((n * d,), MASKED, dtype=torch.uint8, device="cuda")
                n_c, n_l = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
                out = torch.full_like(Q[0], float("nan"))
                outs, seen = torch.full_like(Q, float("nan")), []
                if not callback:
                    steps, left = fdd.fdd_decode_block(ctx, [forkset], layers, d, [list(x) for x in Q], [list(x) for x in K], [list(x) for x in V],
                                                       [list(x) for x in outs], list(S), tokens, state, [d], dim ** -0.5, 0, 0.6, 1.0, 0, 1, n_c, n_l)
                else:
                    q, k, v, s = (torch.empty_like(x[0]) for x in (Q, K, V, S))

                    def before_step(user, t, on):
                        seen.append((user, t, on))
                        if t > 0:
                            outs[t - 1].copy_(out)
                        out.fill_(float("nan"))
                        for buffer, made in ((q, Q), (k, K), (v, V), (s, S)):
                            buffer.copy_(made[t])

                    hook = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p)(before_step)
                    n_steps, n_masked = ctypes.c_int(0), ctypes.c_int(0)
                    rc = fdd.lib().fdd_decode_block(
                        ctx, fdd.ptr_array([forkset]), 1, layers, d, 1, fdd.ptr_array(list(q)), fdd.ptr_array(list(k)), fdd.ptr_array(list(v)),
                        fdd.ptr_array(list(out)), fdd.ptr_array([s]), tokens.data_ptr(), state.data_ptr(), fdd.i32_array([d]), dim ** -0.5, 0,
                        0.6, 1.0, 0, 1, n_c.data_ptr(), n_l.data_ptr(), ctypes.byref(n_steps), ctypes.byref(n_masked),
                        ctypes.cast(hook, ctypes.c_void_p), ctypes.c_void_p(77), ctypes.c_void_p(stream.cuda_stream))
                    assert rc == fdd.FDD_OK
                    steps, left = n_steps.value, n_masked.value
                    if len(seen) == steps:                 # (the step behind the last one is issued ahead, unless the steps ran out)
                        outs[steps - 1].copy_(out)
                    assert [x[1] for x in seen] == list(range(len(seen))) and len(seen) in (steps, steps + 1)
                    assert all(x[0] == 77 and x[2] == stream.cuda_stream for x in seen)
                fdd.fdd_poll_status(ctx)
                return steps, left, tokens.cpu(), state.cpu(), n_l.cpu(), outs, sk.cpu(), sv.cpu()
        finally:
            fdd.fdd_destroy(ctx)

    ref, got = decode(False), decode(True)
    assert got[:2] == ref[:2] and got[1] == 0 and 2 <= got[0] < d
    for a, b in zip(got[2:5], ref[2:5]):
        assert torch.equal(a, b)
    written = ~torch.isnan(ref[5])
    assert torch.equal(~torch.isnan(got[5]), written)
    pu.assert_attention_close(got[5][written].float().cpu().numpy().astype(np.float64), ref[5][written].float().cpu().numpy().astype(np.float64))
    for a, b, made in zip(got[6:], ref[6:], (K, V)):       # (the callback's buffers hold the K/V of the step issued ahead)
        assert torch.equal(b, made[ref[0] - 1].transpose(2, 3).cpu())
        assert torch.equal(a, made[min(got[0], d - 1)].transpose(2, 3).cpu())


@pytest.mark.parametrize("shared", ["out in the logits", "tokens in out", "state in out", "counts in out", "tokens in q", "state in the suffix"])
def test_library_block_loop_where_attention_and_unmasking_share_memory(shared):
    # Attention and unmasking of a step run side by side only where neither writes what the other reads or writes: the
    # result is that of the calls made one by one.
    hq, hkv, dim, vocab, n, d, prefix = 16, 2, 128, 2048, 3, 16, 1000

    def decode(by_library):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(10)
        normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
        ctx = fdd.fdd_create(hq, hkv, dim, vocab, 1, 0, d, n, fdd.FDD_LOGITS_BF16)
        try:
            pk, pv = normal(hkv, prefix, dim), normal(hkv, prefix, dim)
            sk, sv = (torch.zeros((n, hkv, 2 * d, dim), dtype=torch.bfloat16, device="cuda") for _ in range(2))
            q, k, v = normal(n * d * hq * dim), normal(n * d * hkv * dim), normal(n * d * hkv * dim)
            logits = 2.0 * normal(n * d, vocab)
            out = torch.zeros_like(q)
            tokens = torch.full((n * d,), vocab - 1, dtype=torch.int32, device="cuda")
            state = torch.full((n * d,), MASKED, dtype=torch.uint8, device="cuda")
            n_c, n_l = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
            if shared == "out in the logits":
                out = logits.view(-1)[:q.numel()]
            elif shared == "tokens in out":
                tokens = out.view(torch.int32)[64:64 + n * d]
            elif shared == "state in out":
                state = out.view(torch.uint8)[4096:4096 + n * d]
            elif shared == "counts in out":
                n_c = out.view(torch.int32)[128:128 + n]
            elif shared == "tokens in q":
                tokens = q.view(torch.int32)[512:512 + n * d]
                tokens.fill_(vocab - 1)
            else:
                state = sk.view(torch.uint8)[0, 0, d + 3, :n * d]
                state.fill_(MASKED)
            forkset = fdd.fdd_fork(ctx, [pk], [pv], None, prefix, prefix, n, [11, 12, 13], [sk], [sv], 2 * d)
            fdd.fdd_kv_commit(ctx, [forkset], 0, k, v, [d], 1)
            if shared == "state in out":                   # (the first step's attention writes the states that it starts from)
                state.fill_(MASKED)
            if by_library:
                fdd.fdd_decode_block(ctx, [forkset], 1, d, [[q]], [[k]], [[v]], [[out]], [logits], tokens, state, [d], dim ** -0.5, 0, 0.9, 0.7,
                                     0, 0, n_c, n_l)
            else:
                through = False
                for t in range(d):
                    fdd.fdd_block_attn_gated(ctx, [forkset], 0, q, k, v, out, [d], dim ** -0.5, 0, n_l if t else None)
                    fdd.fdd_unmask(ctx, [forkset], logits, tokens, state, [d], 0.9, 0.7, 0, t, n_c, n_l, None)
                    if through:                            # (the library has issued this step before it knew)
                        break
                    through = int(n_l.sum()) == 0
            fdd.fdd_poll_status(ctx)
            return [x.clone() for x in (tokens, state, n_c, n_l, out, logits, q, sk)]
        finally:
            fdd.fdd_destroy(ctx)

    for a, b in zip(decode(True), decode(False)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
