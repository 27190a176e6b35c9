"""Parity of the CUDA library with the CPU oracle at the full sizes of the five workloads, in the launch
configuration the benchmark times (CUDA graphs on).  Contexts too long to prefill on the CPU are injected:
the same seeded recurrent state, conv window and KV rows are given to both sides (prefill itself is compared
on the small configurations).  Every comparison is round by round: candidates, argmax, accept length,
emitted tokens bit-exact where the oracle's margin exceeds 1e-2, logits within 2e-2, states within 1e-3."""
import numpy as np
import pytest

import hs_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import oracle
    from paper_2605_01106_b200 import build, binding
    build.build()
    import harness
    return dict(torch=torch, oracle=oracle, hs=binding, harness=harness)


_W = {}


def make(env, name, batch, max_k, cap, checked, ctx_lens, small_init="jitter", flags=0):
    s = hi.CONFIGS[name]
    if (name, small_init) not in _W:
        _W.clear()                                     # one large blob at a time
        _W[(name, small_init)] = hi.make_weights(s, 0, small_init)
    blob, table = _W[(name, small_init)]
    eng = env["hs"].Engine(s, blob, max_batch=batch, max_k=max_k, kv_capacity=cap, flags=env["hs"].HS_FLAG_GRAPHS | flags)
    model = env["oracle"].Model(s, blob, table, cap)
    seqs = []
    for b in range(batch):
        q = model.new_seq() if b in checked else None
        pending = int(hi.make_prompt(s.V, 1, seq=1000 + b)[0])
        env["harness"].inject_context(eng, q, s, b, int(ctx_lens[b]), pending)
        seqs.append(q)
    eng.set_batch(batch)
    return s, eng, model, seqs


def test_cfg2_full_size_all_k(env):
    s, eng, model, seqs = make(env, "cfg2_0p5b", 1, 8, 640, {0}, [512])
    rep = None
    for k, rounds in ((1, 2), (2, 3), (4, 2), (8, 1)):
        forced = [hi.forced_accept(k, rounds, seq=k)]
        rep = env["harness"].run_rounds(eng, seqs, s, k, rounds, forced=forced, rep=rep)
    print(rep)
    assert eng.device_status() == 0 and rep.rounds == 8


def test_cfg2_full_size_real_acceptance(env):
    s, eng, model, seqs = make(env, "cfg2_0p5b", 1, 2, 600, {0}, [512])
    rep = env["harness"].run_rounds(eng, seqs, s, 2, 3)
    print(rep)
    assert eng.device_status() == 0


@pytest.mark.parametrize("name,ctx", [("cfg2_0p5b", 512), ("cfg4_seq", 1024)])
def test_full_size_rollback_by_replay(env, name, ctx):
    s, eng, model, seqs = make(env, name, 2, 4, ctx + 100, {0, 1}, [ctx, ctx - 37], flags=env["hs"].HS_FLAG_REPLAY)
    rep = env["harness"].run_rounds(eng, seqs, s, 2, 2, forced=[[0, 2], [1, 0]])
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 2, forced=[[4, 1], [2, 3]], rep=rep)
    print(rep)
    assert eng.device_status() == 0 and rep.rounds == 4


def test_cfg2_attention_geometries(env):
    # the split of the KV cache over CTAs (keys per tile x tiles per CTA) is a launch-time choice: every
    # setting, including several tiles per CTA (running softmax), ragged last tiles and more than one
    # cluster per sequence, must reproduce the oracle on two sequences of different context length
    s, eng, model, seqs = make(env, "cfg2_0p5b", 2, 4, 1024, {0, 1}, [700, 333])
    with pytest.raises(RuntimeError):
        eng.set_attn_geometry(40, 1)
    rep = None
    for chunk, tiles in ((32, 2), (32, 4), (48, 2), (64, 2), (64, 8), (96, 1), (128, 2), (128, 1), (0, 0)):
        seqs = [model.new_seq(), model.new_seq()]
        for b, n in enumerate((700, 333)):
            env["harness"].inject_context(eng, seqs[b], s, b, n, 11 + b)
        eng.set_batch(2)
        eng.set_attn_geometry(chunk, tiles)
        rep = env["harness"].run_rounds(eng, seqs, s, 4, 1, forced=[[2], [4]], rep=rep)
        assert eng.device_status() == 0, (chunk, tiles)
    print(rep)
    assert rep.rounds == 9


def test_cfg2_projection_kernel_choices(env):
    # which kernel a projection runs on is a matter of its activation-row count (CUDA cores up to 3 rows, the
    # warp-level tensor path, tcgen05 from a threshold on): every choice must reproduce the oracle.  Threshold 17 keeps
    # 6 and 10 rows on the warp-level path (one and two groups of eight rows), 2 sends even the two-row draft steps
    # through tcgen05 (16- and 32-row tiles, K split over clusters), 0 restores the automatic threshold.
    s, eng, model, seqs = make(env, "cfg2_0p5b", 2, 8, 700, {0, 1}, [512, 77])
    with pytest.raises(RuntimeError):
        eng.set_option(eng.OPT_TC_MIN_ROWS, 18)
    rep = None
    try:
        for thr, ks in ((17, (2, 4)), (2, (0, 2, 8)), (0, (1, 4))):
            eng.set_option(eng.OPT_TC_MIN_ROWS, thr)
            for k in ks:
                forced = [hi.forced_accept(k, 1, seq=thr + k + b) for b in range(2)]
                rep = env["harness"].run_rounds(eng, seqs, s, k, 1, forced=forced, rep=rep)
                assert eng.device_status() == 0, (thr, k)
    finally:
        eng.set_option(eng.OPT_TC_MIN_ROWS, 0)
    print(rep)
    assert rep.rounds == 7


@pytest.mark.parametrize("name,L", [("cfg2_0p5b", 2), ("cfg4_seq", 4)])
@pytest.mark.parametrize("batch,k", [(4, 1), (7, 1), (16, 2), (17, 3), (33, 4), (40, 4)])
def test_projections_and_packed_mixers_by_rows(env, monkeypatch, name, L, batch, k):
    # tcgen05 projections of 4 .. 200 activation rows on the 1024-wide layers: residual ones in tiles of 64 weight rows (up to 17
    # rows) and of 128, 16 .. 128 rows per tile, K split over clusters whose last rank finishes fewer rows or none; the mixers of
    # the draft steps (4 .. 40 rows) and the DeltaNet layers (below 192 rows) pack the out-projection's operand themselves
    s = hi.CONFIGS[name].replace(L=L, V=2048)
    monkeypatch.setitem(hi.CONFIGS, "small", s)
    _W.pop(("small", "jitter"), None)
    _, eng, model, seqs = make(env, "small", batch, k, 96, {0, batch // 2, batch - 1}, [20 + 3 * (b % 9) for b in range(batch)])
    _W.pop(("small", "jitter"), None)
    forced = [hi.forced_accept(k, 2, seq=b) for b in range(batch)]
    rep = env["harness"].run_rounds(eng, seqs, s, k, 2, forced=forced)
    print(rep)
    assert rep.rounds == 2 and eng.device_status() == 0


@pytest.mark.parametrize("name,plan,batch,on_tcgen05", [
    ("cfg1_tiny", "component", 3, False), ("cfg1_tiny", "component", 4, True),
    ("cfg1_tiny", "full", 5, False), ("cfg1_tiny", "full", 6, True), ("cfg1_tiny", "layerskip33", 4, False),
    ("test_seq", "component", 4, True), ("test_seq", "full", 4, False), ("test_seq", "full", 5, True)])
def test_row_threshold_of_draft_steps(env, name, plan, batch, on_tcgen05):
    # a draft step runs on tcgen05 from 4 rows on where its mixers pack the out-projection's operand, later where the plan keeps
    # attention: there is at least one packing kernel more (the embedding's) than with the threshold out of reach
    s = hi.CONFIGS[name]
    eng = env["hs"].Engine(s, np.zeros(hi.blob_layout(s)[1], np.uint8), max_batch=batch, max_k=1, kv_capacity=64)
    eng.set_draft_plan(hi.draft_plan(s, plan))
    for b in range(batch):
        eng.set_context(b, 20, 1)
    eng.set_batch(batch)
    count = {}
    try:
        for threshold in (0, 2, 17):
            eng.set_option(eng.OPT_TC_MIN_ROWS, threshold)
            before = eng.launch_count()
            eng.draft(1)
            count[threshold] = eng.launch_count() - before
    finally:
        eng.set_option(eng.OPT_TC_MIN_ROWS, 0)
    assert count[2] > count[17] and count[0] == count[2 if on_tcgen05 else 17], count
    assert eng.device_status() == 0


def test_row_threshold_belongs_to_the_handle(env):
    # a threshold set on one handle reaches neither one that is there already nor one that is made afterwards
    s = hi.CONFIGS["cfg1_tiny"]

    def engine():
        e = env["hs"].Engine(s, np.zeros(hi.blob_layout(s)[1], np.uint8), max_batch=4, max_k=1, kv_capacity=64)
        for b in range(4):
            e.set_context(b, 20, 1)
        e.set_batch(4)
        return e

    def launches(e):
        before = e.launch_count()
        e.draft(1)
        return e.launch_count() - before

    first, second = engine(), engine()
    automatic = launches(first)
    second.set_option(second.OPT_TC_MIN_ROWS, 17)
    try:
        assert launches(second) < automatic and launches(first) == automatic and launches(engine()) == automatic
    finally:
        second.set_option(second.OPT_TC_MIN_ROWS, 0)
    assert launches(second) == automatic


def test_streaming_attention_edge_cases(env):
    # the streaming form (128-key tiles walked through a ring of buffers, warp-local running softmax, ranges merged by the last
    # CTA to arrive) on the small sequential stack, where attention is a launch of its own: contexts that end exactly on
    # a tile boundary (the new rows then form a ninth key group), one key short of and one past it, a single short
    # range, several tiles per CTA, one and two 16-row query tiles (k = 4: 10 rows, k = 8: 18 rows)
    lens = [1152, 1151, 1153, 640, 77, 1279]
    s, eng, model, seqs = make(env, "test_seq", len(lens), 8, 1500, set(range(len(lens))), lens)
    rep = None
    for tiles, k in ((-1, 4), (-2, 8), (-4, 4), (-16, 8), (-3, 1)):
        eng.set_attn_geometry(128, tiles)
        forced = [hi.forced_accept(k, 1, seq=40 + b - tiles) for b in range(len(lens))]
        rep = env["harness"].run_rounds(eng, seqs, s, k, 1, forced=forced, rep=rep)
        assert eng.device_status() == 0, (tiles, k)
    with pytest.raises(RuntimeError):
        eng.set_attn_geometry(64, -2)
    print(rep)
    assert rep.rounds == 5


@pytest.mark.parametrize("tiles,k,lens", [
    (-1, 4, [3500, 3201, 3072]),        # a full tile of query rows: 28 ranges of one tile, sixteen warps in two groups
    (-2, 4, [3073, 2944, 300]),         # 13 ranges of two tiles: eight warps
    (-16, 1, [1279, 900, 700]),         # a packed tile: a whole cache of 6 to 10 tiles, sixteen warps
    (-2, 1, [1279, 640, 77])])          # several ranges: eight warps
def test_streaming_attention_by_warps(env, tiles, k, lens):
    s, eng, model, seqs = make(env, "test_seq", len(lens), k, max(lens) + 64, set(range(len(lens))), lens)
    eng.set_attn_geometry(128, tiles)
    rep = env["harness"].run_rounds(eng, seqs, s, k, 2, forced=[hi.forced_accept(k, 2, seq=70 + b) for b in range(len(lens))])
    print(rep)
    assert rep.rounds == 2 and eng.device_status() == 0


@pytest.mark.parametrize("lens,checked,ks", [
    ([7000, 6913], {0, 1}, (4, 3, 2, 1, 0)),                    # 28 ranges of two tiles, merged two rows per thread from 9 rows on
    ([1600 - 53 * (b % 29) for b in range(100)], {0, 1, 50, 99}, (3, 2, 0))])       # equal shares
def test_streaming_attention_of_wide_heads(env, monkeypatch, lens, checked, ks):
    # 128-wide heads, 4 .. 20 query rows per KV head: packed, full, full and packed query tiles
    s = hi.CONFIGS["cfg2_0p5b"].replace(L=1, V=2048)
    monkeypatch.setitem(hi.CONFIGS, "wide", s)
    _W.pop(("wide", "jitter"), None)
    _, eng, model, seqs = make(env, "wide", len(lens), max(ks), max(lens) + 64, checked, lens)
    _W.pop(("wide", "jitter"), None)
    rep = None
    for k in ks:
        forced = [hi.forced_accept(k, 1, seq=20 + b + k) for b in range(len(lens))]
        rep = env["harness"].run_rounds(eng, seqs, s, k, 1, forced=forced, rep=rep)
        assert eng.device_status() == 0, k
    print(rep)
    assert rep.rounds == len(ks)


@pytest.mark.parametrize("hd,qh,k,tiles", [(64, 8, 4, -16), (64, 8, 4, -17), (64, 8, 7, -2), (64, 8, 7, -17), (128, 8, 4, -3), (128, 8, 7, -16)])
def test_streaming_attention_two_query_tiles(env, monkeypatch, hd, qh, k, tiles):
    # two tiles of query rows, the second one packed (20 rows) or full (32), with a fixed number of tiles per CTA: up to 16 the products
    # of a range run on in the same accumulators, beyond that every tile has its own
    name = "test_seq_h%d_q%d" % (hd, qh)
    s = hi.CONFIGS["test_seq"].replace(qh=qh, hd=hd)
    monkeypatch.setitem(hi.CONFIGS, name, s)
    lens = [2303, 2176, 2049, 5]
    _, eng, model, seqs = make(env, name, len(lens), k, 2400, set(range(len(lens))), lens)
    eng.set_attn_geometry(128, tiles)
    rep = env["harness"].run_rounds(eng, seqs, s, k, 2, forced=[hi.forced_accept(k, 2, seq=30 + b) for b in range(len(lens))])
    print(rep)
    assert rep.rounds == 2 and eng.device_status() == 0


@pytest.mark.parametrize("qh,ks", [(4, (8, 4, 1)), (8, (7,))])
def test_streaming_attention_in_equal_shares(env, monkeypatch, qh, ks):
    # more than 16 rounds' worth of tiles (2600 by the longest of 100 caches): one CTA per SM with an equal share of the tiles of all
    # caches, which starts and ends inside them; caches of many tiles, of one (full, one key short, one key over) and of a few keys,
    # one query tile (plain, packed) and two (second one packed, plain)
    s = hi.CONFIGS["test_seq"].replace(qh=qh)
    monkeypatch.setitem(hi.CONFIGS, "test_seq_q%d" % qh, s)
    sizes, batch, checked = (1600, 128, 127, 129, 5, 640, 1599, 1024), 100, {0, 1, 2, 3, 4, 38, 95, 99}
    lens = [sizes[b % 8] if b % 3 else 1600 - b for b in range(batch)]
    lens[:5] = [1600, 128, 127, 129, 5]
    _, eng, model, seqs = make(env, "test_seq_q%d" % qh, batch, max(ks), 1700, checked, lens)
    rep = None
    for k in ks:
        forced = [hi.forced_accept(k, 1, seq=40 + b + k) for b in range(batch)]
        rep = env["harness"].run_rounds(eng, seqs, s, k, 1, forced=forced, rep=rep)
        assert eng.device_status() == 0, k
    assert rep.rounds == len(ks)


def test_streaming_attention_in_equal_shares_of_a_draft(env):
    # a draft that keeps attention reads its own rows behind the cache (one more per step), here in equal shares: step i starts its
    # new row at kv_len + i, on both sides of a tile boundary
    lens = [1600 - 37 * (b % 31) for b in range(100)]
    lens[:6] = [1535, 1534, 1533, 1536, 127, 128]
    s, eng, model, seqs = make(env, "test_seq", len(lens), 4, 1700, {0, 1, 2, 3, 4, 5, 57, 99}, lens)
    plan = hi.draft_plan(s, "full")
    eng.set_draft_plan(plan)
    model.set_draft_plan(plan)
    forced = [hi.forced_accept(4, 2, seq=b) for b in range(len(lens))]
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 2, forced=forced)
    print(rep)
    assert rep.rounds == 2 and eng.device_status() == 0


def test_streaming_attention_in_equal_shares_of_many_sequences(env):
    # more sequences than a block has threads: a thread counts the tiles of several; shares of 16 tiles, most of them over many caches
    batch, checked = 600, {0, 1, 2, 255, 256, 511, 512, 598, 599}
    lens = [250 - (7 * b) % 245 for b in range(batch)]
    lens[:3], lens[598:] = [128, 129, 250], [127, 250]
    s, eng, model, seqs = make(env, "test_seq", batch, 1, 300, checked, lens)
    forced = [hi.forced_accept(1, 2, seq=b) for b in range(batch)]
    rep = env["harness"].run_rounds(eng, seqs, s, 1, 2, forced=forced)
    print(rep)
    assert rep.rounds == 2 and eng.device_status() == 0


@pytest.mark.parametrize("form", ["fixed tiles", "equal shares"])
def test_streaming_attention_control_words_out_of_range(env, form):
    # a bad cache length of one sequence in the streaming form, with a fixed number of tiles per CTA and in equal shares (where a CTA
    # goes on with the next cache of its share): the status word names the error however far beyond the cache the length lies - the
    # grid has no CTA for the last range of such a cache -, guard bytes stay intact and the other sequences reproduce the oracle.
    # (Sequence 0 of many: even an unchecked access would stay inside the cache.)
    if form == "fixed tiles":
        cap, lens, checked = 1500, [700, 1151, 640, 77, 1279, 128], {1, 2, 3, 4, 5}
    else:
        cap, lens, checked = 1700, [1600 - 53 * (b % 29) for b in range(100)], {1, 2, 50, 99}
    s, eng, model, seqs = make(env, "test_seq", len(lens), 4, cap, checked, lens)
    if form == "fixed tiles":
        eng.set_attn_geometry(128, -2)
    rep = None
    for value, want in ((cap - 2, -3), (cap + 1000, -3), (3 * cap, -3), (2 ** 31 - 3, -3), (-5, -7)):
        eng.poke_control(0, eng.CTRL_KV_LEN, value)
        forced = [hi.forced_accept(4, 1, seq=b - want) for b in range(len(lens))]
        rep = env["harness"].run_rounds(eng, seqs, s, 4, 1, forced=forced, rep=rep)
        assert eng.device_status() == want, value
        eng.clear_status()
    print(rep)
    assert rep.rounds == 5


@pytest.mark.parametrize("qh,k", [(8, 4), (4, 4), (4, 1)])
def test_streaming_attention_long_shares_stay_exact(env, qh, k):
    # 250 tiles of 128 keys per CTA (equal shares), every cached V row of a KV head the same: whatever the probabilities are, the
    # attention's output is that row.  The tensor path truncates when it adds to an accumulator (2^-26 of the sum per MMA on
    # average), so a chain over a whole share would leave the output short by 2e-6 to 4e-6.  A tile's products in accumulators of
    # their own lose at most 2 * 2^-26; the out-projection's factor for its own chain of 8 MMAs adds 8 * 2^-26 here, where a sum has
    # one term: below 2e-7 together, 5e-7 allowed.  One-layer model: Mamba branch and MLP zero, W_o and the LM head copy, the
    # last 256 dimensions carry the embedding (1), by which the logits are divided to take the final norm out.
    torch = env["torch"]
    hd, kvh, batch, T = 64, 2, 9, k + 1
    n_o, n = qh * hd, 2056 * 128
    d = n_o + 256
    s = hi.CONFIGS["cfg1_tiny"].replace(L=1, d=d, V=d, qh=qh, kvh=kvh, hd=hd, ff=256)
    table, nbytes = hi.blob_layout(s)
    blob = np.zeros(nbytes, np.uint8)
    rng = np.random.default_rng(5)

    def put(layer, tid, a):
        off, dims, dt = table[(layer, tid)]
        assert a.shape == tuple(dims)
        a = torch.from_numpy(np.ascontiguousarray(a, np.float32))
        a = a.to(torch.bfloat16).view(torch.uint8).numpy() if dt == "bf16" else a.numpy().view(np.uint8)
        blob[off:off + a.nbytes] = a.reshape(-1)

    c = torch.from_numpy(rng.uniform(0.5, 1.5, (kvh, hd)).astype(np.float32)).to(torch.bfloat16)
    eye = np.eye(d, dtype=np.float32)
    put(-1, hi.G_EMBED, np.concatenate([np.zeros((d, n_o)), np.ones((d, 256))], 1))
    put(-1, hi.G_LM_HEAD, eye)
    put(-1, hi.G_FINAL_NORM, np.ones(d))
    put(0, hi.T_NORM1, np.full(d, np.sqrt(256 / d + s.eps)))
    put(0, hi.T_NORM2, np.ones(d)); put(0, hi.T_GNORM, np.ones(s.d_inner))
    w = np.zeros(table[(0, hi.T_W_IN)][1], np.float32)
    q0 = w.shape[0] - (qh + 2 * kvh) * hd
    w[q0:q0 + n_o, n_o:] = rng.normal(0.0, 0.07, (n_o, 256))
    w[q0 + n_o + kvh * hd:, n_o] = c.float().numpy().reshape(-1)
    put(0, hi.T_W_IN, w)
    put(0, hi.T_W_O, eye[:, :n_o])
    eng = env["hs"].Engine(s, blob, max_batch=batch, max_k=k, kv_capacity=n + 16)
    kv = eng.t_kv[:2 * 2 * batch * kvh * (n + 16) * hd].view(torch.bfloat16).view(2, batch, kvh, n + 16, hd)
    kv[0].normal_(generator=torch.Generator(device=eng.device).manual_seed(7))
    kv[1].copy_(c.to(eng.device)[None, :, None, :].expand(batch, kvh, n + 16, hd))
    for b in range(batch):
        eng.set_context(b, n, 1)
    eng.set_batch(batch)
    eng.verify(k, torch.ones((batch, T), dtype=torch.int32, device=eng.device))
    lg = eng.get_logits(batch * T).astype(np.float64)
    assert eng.device_status() == 0 and eng.check_guards()
    o = lg[:, :n_o] / lg[:, n_o:].mean(1, keepdims=True)
    want = c.double().numpy()[np.arange(qh) // (qh // kvh)].reshape(1, n_o)
    err = (o / want - 1).reshape(batch, T, qh, hd)
    print("shortfall of the output: mean %.2e, by head %s" % (-err.mean(), -err.mean((0, 1, 3))))
    assert abs(err.mean()) <= 5e-7 and np.abs(err.mean((0, 1, 3))).max() <= 5e-7
    assert np.abs(err).max() <= 2.0 ** -14              # operands as bf16 head and remainder: 2^-17 each


@pytest.mark.parametrize("name,geometry", [("test_seq", (0, 0)), ("test_seq", (64, 4)), ("cfg1_tiny", (0, 0)), ("cfg1_tiny", (64, 4))])
def test_control_words_near_the_integer_limit(env, name, geometry):
    # a cache length to which nothing can be added: reported, not used, in the lean and the general form, alone and beside a mixer
    lens = [200, 333, 77]
    s, eng, model, seqs = make(env, name, len(lens), 4, 512, {1, 2}, lens)
    eng.set_attn_geometry(*geometry)
    rep = None
    for value in (2 ** 31 - 1, 2 ** 31 - 4):
        eng.poke_control(0, eng.CTRL_KV_LEN, value)
        rep = env["harness"].run_rounds(eng, seqs, s, 4, 1, forced=[hi.forced_accept(4, 1, seq=b) for b in range(len(lens))], rep=rep)
        assert eng.device_status() == -3, value
        eng.clear_status()
    assert rep.rounds == 2


def test_streaming_attention_batched_parallel_hybrid(env):
    # a batch large enough that the verify attention of the parallel hybrid runs as its own launch in the streaming form
    # (chosen automatically); three sequences carry their context on both sides, the others run beside them
    lens = [1152, 1151, 640] + [1000 + 7 * b for b in range(21)]
    s, eng, model, seqs = make(env, "cfg1_tiny", len(lens), 4, 1400, {0, 1, 2}, lens)
    forced = [hi.forced_accept(4, 2, seq=b) for b in range(len(lens))]
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 2, forced=forced)
    forced = [hi.forced_accept(2, 2, seq=50 + b) for b in range(len(lens))]
    rep = env["harness"].run_rounds(eng, seqs, s, 2, 2, forced=forced, rep=rep)
    print(rep)
    assert eng.device_status() == 0 and rep.rounds == 4


def test_cfg4_sequential_full_size(env):
    s, eng, model, seqs = make(env, "cfg4_seq", 1, 4, 1100, {0}, [1024])
    rep = env["harness"].run_rounds(eng, seqs, s, 2, 2, forced=[hi.forced_accept(2, 2, seq=1)])
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 1, forced=[hi.forced_accept(4, 1, seq=2)], rep=rep)
    print(rep)
    assert eng.device_status() == 0


def test_cfg3_3b_batch1(env):
    # perturbed small parameters (norm weights, D, conv bias): a kernel that dropped one of them at this shape
    # (N = 256, 80 heads, 20 query heads) would be noticed
    s, eng, model, seqs = make(env, "cfg3_3b", 1, 4, 2100, {0}, [2048])
    rep = env["harness"].run_rounds(eng, seqs, s, 2, 1, forced=[[1]])
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 1, forced=[[2]], rep=rep)
    print(rep)
    assert eng.device_status() == 0


def test_cfg3_3b_batch8_two_checked(env):
    s, eng, model, seqs = make(env, "cfg3_3b", 8, 4, 2100, {0, 5}, [2048] * 8)
    forced = [hi.forced_accept(4, 1, seq=b) for b in range(8)]
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 1, forced=forced)
    forced = [hi.forced_accept(2, 1, seq=20 + b) for b in range(8)]
    rep = env["harness"].run_rounds(eng, seqs, s, 2, 1, forced=forced, rep=rep)
    print(rep)
    assert eng.device_status() == 0


def test_cfg5_batch64_ragged_sampled(env):
    # 64 sequences with contexts uniform in [4096, 16384]; four of them carry a full seeded context on both
    # sides and are compared, the others run beside them with their own accept pattern (ragged rollback)
    s = hi.CONFIGS["cfg5_b64"]
    lens = hi.context_lengths(64, 4096, 16384)
    checked = {0, 17, 38, 63}
    s, eng, model, seqs = make(env, "cfg5_b64", 64, 4, 16384 + 32, checked, lens)
    forced = [hi.forced_accept(4, 2, seq=b) for b in range(64)]
    rep = env["harness"].run_rounds(eng, seqs, s, 4, 2, forced=forced)
    print(rep, sorted(set(int(x) for x in lens))[:3])
    for b in range(64):
        kv, _ = eng.get_context(b)
        assert kv == lens[b] + int((np.array(forced[b]) + 1).sum())
    assert len(rep.n_hist) >= 2 and eng.device_status() == 0


def test_cfg5_batch64_two_sequences_128_tokens(env):
    # the long run of the batch-64 workload: 64 ragged sequences decode 128 tokens each (k = 4, seeded accept
    # pattern, about 48 rounds); two of them carry their full context on the CPU side as well and are compared
    # round by round over the whole generation, states every eighth round
    s = hi.CONFIGS["cfg5_b64"]
    lens = hi.context_lengths(64, 4096, 16384)
    rounds = 48
    s, eng, model, seqs = make(env, "cfg5_b64", 64, 4, 16384 + 5 * (rounds + 2), {5, 41}, lens)
    forced = [hi.forced_accept(4, rounds, seq=100 + b) for b in range(64)]
    rep = env["harness"].run_rounds(eng, seqs, s, 4, rounds, forced=forced, check_states_every=8)
    print(rep)
    assert rep.tokens >= 2 * 110 and eng.device_status() == 0
    for b in (5, 41):
        kv, _ = eng.get_context(b)
        assert kv == lens[b] + int((np.array(forced[b]) + 1).sum())


@pytest.mark.parametrize("name,k,ctx", [("cfg1_tiny", 8, 255), ("cfg1_tiny", 8, 129), ("test_seq", 8, 2000)])
def test_lean_attention_with_several_row_tiles(env, name, k, ctx):
    # 17 and more query rows per KV head in the latency-lean form: several clusters of 16 rows each, the last one ragged
    # (two query heads per KV head x 9 positions = 18 rows), of which only the first appends to the cache
    s, eng, model, seqs = make(env, name, 1, k, ctx + 64, {0}, [ctx])
    rep = env["harness"].run_rounds(eng, seqs, s, k, 3, forced=[[8, 3, 0]])
    print(rep)
    assert eng.device_status() == 0


@pytest.mark.parametrize("name,batch,k,ctx", [
    ("cfg1_tiny", 1, 4, 1019), ("cfg1_tiny", 1, 4, 1020),       # 1024 keys: lean beside the mixer; 1025: lean, a launch of its own
    ("cfg1_tiny", 1, 4, 2299), ("cfg1_tiny", 1, 4, 2300),       # 2304 keys: the longest lean cache; 2305: general form beside the mixer
    ("cfg1_tiny", 3, 4, 2300), ("cfg1_tiny", 20, 2, 100),       # 114 tiles of 128 keys: streaming; 640 mixer blocks: apart, lean
    ("cfg1_tiny", 38, 2, 100), ("cfg1_tiny", 26, 4, 200),       # more than 4 lean CTAs per SM: general; 104 tiles, two per cache: streaming
    ("cfg2_0p5b", 1, 2, 2301)])                                 # 288 keys per CTA at a head dimension of 128
def test_attention_form_boundaries(env, name, batch, k, ctx):
    s, eng, model, seqs = make(env, name, batch, k, ctx + 32, {0}, [ctx] * batch)
    rep = env["harness"].run_rounds(eng, seqs, s, k, 1, forced=[hi.forced_accept(k, 1, seq=b) for b in range(batch)])
    print(rep)
    assert eng.device_status() == 0


@pytest.mark.parametrize("name", ["cfg1_tiny", "test_seq"])
def test_mixer_instances_by_positions(env, name):
    # 4 and 5 positions run in the instance for 5, 6 in the one for 9; two sequences, their rows beside each other
    s, eng, model, seqs = make(env, name, 2, 5, 160, {0, 1}, [70, 33])
    rep = None
    for k in (3, 4, 5):
        rep = env["harness"].run_rounds(eng, seqs, s, k, 2, forced=[hi.forced_accept(k, 2, seq=b + k) for b in range(2)], rep=rep)
    print(rep)
    assert eng.device_status() == 0 and rep.rounds == 6


@pytest.mark.parametrize("name,batch,k,ctx,apart", [
    ("cfg2_0p5b", 1, 8, 1000, False), ("cfg2_0p5b", 3, 2, 700, False),
    ("cfg2_0p5b", 3, 4, 700, True),          # 96 keys per CTA and two row tiles: one block fits an SM, 3.2 rounds of them
    ("cfg2_0p5b", 4, 8, 100, True), ("cfg3_3b", 1, 4, 700, True), ("cfg3_3b", 1, 4, 250, False)])
def test_mixer_and_attention_share_a_launch_while_blocks_fit(env, name, batch, k, ctx, apart):
    s = hi.CONFIGS[name].replace(L=1, V=512)
    eng = env["hs"].Engine(s, np.zeros(hi.blob_layout(s)[1], np.uint8), max_batch=batch, max_k=k, kv_capacity=ctx + 32)
    for b in range(batch):
        eng.set_context(b, ctx, 1)
    eng.set_batch(batch)
    eng.draft(k)
    eng.profile(True)
    eng.verify(k)
    prof = eng.profile_read()
    eng.profile(False)
    eng.accept_rollback()
    assert (prof["attention"][1] == 1) == apart and eng.device_status() == 0, prof
