"""Prompts longer than one verify pass: the wide prefill path against the CPU oracle at the sizes where it can go wrong
(edges of the 8-position scan tiles, the 16-row conv tiles, the 64-position attention tiles; prompts of one to three
positions beyond a conv window; a batch that needs more than one pass; a prompt appended to a context; every size class of
the scans; every form of the two-CTA projections), sequences beside one that is not finite, and the precision of its sums."""
import numpy as np
import pytest

import hs_inputs as hi

pytestmark = pytest.mark.gpu

SHAPES = {
    "par64": hi.CONFIGS["cfg1_tiny"],
    "par128": hi.CONFIGS["cfg1_tiny"].replace(N=128, hd=128),
    "par256": hi.CONFIGS["cfg1_tiny"].replace(N=256, H=12, qh=6, kvh=2, hd=128),
    "seq": hi.CONFIGS["test_seq"],
    "seq32": hi.CONFIGS["test_seq"].replace(gdv=32, gh=8, hd=128),
    "seq16": hi.CONFIGS["test_seq"].replace(gh=16),
}


@pytest.fixture(scope="module")
def env():
    import oracle
    from paper_2605_01106_b200 import build, binding
    build.build()
    import harness
    return dict(oracle=oracle, hs=binding, harness=harness)


@pytest.mark.parametrize("name,lens,max_k,flags", [
    ("par64", [65, 1, 16, 129, 7], 4, 0),
    ("par64", [1500, 2, 700, 33], 8, 2),          # two passes; rollback by replay
    ("par128", [64, 63, 130], 2, 1),
    ("par256", [17, 50], 4, 0),
    ("par256", [9], 2, 0), ("par256", [17, 50, 8, 20], 2, 0), ("par256", [17, 50, 8, 20, 11], 2, 1),      # 2, 6 and 5 x 8 rows of the scan per warp
    ("par128", [17, 9, 8, 20, 11], 2, 0), ("par64", [17, 9, 8, 20, 11, 3, 33], 2, 0),
    ("seq", [72, 3, 9, 128, 40], 4, 0),
    ("seq", [1100, 1100], 8, 2),
    ("seq32", [66, 31], 8, 1),
    ("seq16", [9, 17, 8, 30, 5], 2, 0),           # 320 strips of 16 value rows: two rows per lane group
    ("par64", [9, 17, 8, 11, 12, 20, 5, 33, 10, 16, 7, 13], 2, 0),        # 6144 state rows: several scan blocks per SM, four stages
])
def test_wide_prefill_matches_oracle(env, name, lens, max_k, flags):
    s = SHAPES[name]
    blob, table = hi.make_weights(s, 0, "jitter")
    cap = max(lens) + 64
    eng = env["hs"].Engine(s, blob, max_batch=len(lens), max_k=max_k, kv_capacity=cap, flags=flags)
    model = env["oracle"].Model(s, blob, table, cap)
    prompts = [hi.make_prompt(s.V, n, seq=40 + b) for b, n in enumerate(lens)]
    seqs = [model.new_seq() for _ in lens]
    for q, p in zip(seqs, prompts):
        q.prefill(p)
    eng.prefill(prompts)
    env["harness"].compare_states(eng, seqs, s, kv_rows=None)
    rep = env["harness"].run_rounds(eng, seqs, s, max_k, 2, forced=[hi.forced_accept(max_k, 2, seq=b) for b in range(len(lens))])
    # the next turn of a conversation: prompts appended behind what every sequence holds
    more = [hi.make_prompt(s.V, 11 + 2 * b, seq=80 + b) for b in range(len(lens))]
    for q, p in zip(seqs, more):
        q.prefill(p)
    eng.prefill(more)
    env["harness"].compare_states(eng, seqs, s, rep)
    assert eng.device_status() == 0


def test_logits_after_prefill(env):
    # get_logits after a prefill: the positions of the prompt's last chunk of max_k + 1
    s = SHAPES["par64"]
    blob, table = hi.make_weights(s, 0, "jitter")
    eng = env["hs"].Engine(s, blob, max_batch=1, max_k=4, kv_capacity=96)
    model = env["oracle"].Model(s, blob, table, 96)
    prompt = hi.make_prompt(s.V, 48, seq=5)
    eng.prefill([prompt])
    got = eng.get_logits(3)                       # 48 = 9 * 5 + 3
    for i in range(3):
        q = model.new_seq()
        q.prefill(prompt[:45])
        want = q.round(2, cand_in=np.asarray(prompt[45:48], np.int32), forced_n=2, want_logits=True)["logits"][i]
        assert np.abs(got[i] - want).max() <= env["harness"].LOGIT_TOL


@pytest.mark.parametrize("name,lens,max_k", [("par64", [13, 9, 20], 4), ("par128", [3, 30, 8, 12], 2), ("par256", [21, 4, 33], 4), ("seq", [13, 9, 20], 4), ("seq32", [31, 6], 4)])
def test_sequences_of_a_prompt_pass_are_independent(env, name, lens, max_k):
    # sequence 1 consists of a token whose embedding is not finite; the others, whose last partial scan tile lies in front of
    # its rows or whose rows lie behind them, are what they are without it
    s = SHAPES[name]
    blob, table = hi.make_weights(s, 0, "jitter")
    prompts = [hi.make_prompt(s.V, n, seq=40 + b) for b, n in enumerate(lens)]
    bad = next(t for t in range(s.V) if all(t not in p for p in prompts))
    prompts[1] = np.full(lens[1], bad, np.int32)
    off = table[(-1, hi.G_EMBED)][0] + 2 * s.d * bad
    blob[off:off + 2 * s.d].view(np.uint16)[:] = 0x7FC0                # bf16 NaN
    cap = max(lens) + 32
    eng = env["hs"].Engine(s, blob, max_batch=len(lens), max_k=max_k, kv_capacity=cap)
    model = env["oracle"].Model(s, blob, table, cap)
    seqs = [None if b == 1 else model.new_seq() for b in range(len(lens))]
    for q, p in zip(seqs, prompts):
        if q is not None:
            q.prefill(p)
    eng.prefill(prompts)
    env["harness"].compare_states(eng, seqs, s)
    assert eng.device_status() == 0


@pytest.mark.parametrize("d,H,n", [(1024, 32, 70), (1024, 32, 600), (2560, 80, 70), (2560, 80, 300), (2560, 80, 2048), (4096, 64, 1100)])
def test_prompt_projections_are_as_exact_as_their_operands(env, d, H, n):
    # Raw conv inputs of the first layer: in-projection sums of d terms, which depend on the last three tokens only.  bf16 head
    # and remainder hold an activation to at most 2^-18 of itself, 2.45e-6 rms in the sums.  Truncation in tensor memory adds a
    # spread of at most 0.6 * 64 * 2^-26 = 0.57e-6 (64 MMAs per accumulator; 2.52e-6 together, 10 % on top for the sample of
    # about 7000 values) and its mean, -2^-26 of a sum per MMA, is put back (what is left: 15 % of 64 * 2^-26, and the
    # standard error of the slope, 3e-8)
    s = hi.CONFIGS["cfg2_0p5b"].replace(L=1, V=2048, d=d, H=H, ff=512)
    blob, table = hi.make_weights(s, 0, "jitter")
    eng = env["hs"].Engine(s, blob, max_batch=1, max_k=4, kv_capacity=n + 8)
    p = hi.make_prompt(s.V, n, seq=41)
    eng.prefill([p])
    q = env["oracle"].Model(s, blob, table, 8).new_seq()
    q.prefill(p[-3:])
    want = np.asarray(q.conv()[0], np.float64)
    got = eng.export_state(0, 0, env["hs"].STATE_CONV).astype(np.float64)
    slope = (got * want).sum() / (want * want).sum() - 1
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    print(d, n, "slope %.2e error %.2e" % (slope, err))
    assert abs(slope) < 0.35e-6 and err < 2.8e-6 and eng.device_status() == 0


def test_attention_over_a_long_cache_is_as_exact_as_its_operands(env):
    # A prompt behind 4000 imported keys (the same bits on both sides); the attention of the first layer carries the residual
    # stream (embedding small, no mixer, no MLP) that the next layer's conv inputs are made of.  Probabilities, the attention's
    # output and the stream are held as bf16 head and remainder on the way, 2.45e-6 rms each: 4.2e-6 for the three.  One
    # accumulator over all keys would truncate 500 times: 0.6 * 500 * 2^-26 = 4.5e-6 of spread on top, 6.2e-6
    s = hi.CONFIGS["cfg1_tiny"]
    ctx = 4000
    blob, table = hi.make_weights(s, 0, "unit")
    bf = lambda l, t: blob[table[(l, t)][0]:table[(l, t)][0] + 2 * int(np.prod(table[(l, t)][1]))].view(np.uint16)
    bf(0, hi.T_W_OUT)[:] = 0
    bf(0, hi.T_W_DOWN)[:] = 0
    e = bf(-1, hi.G_EMBED)
    e[:] = (hi.bf16_to_f32(e).ravel() * np.float32(2.0 ** -6)).view(np.uint32) >> 16          # an exact shift of the exponent
    eng = env["hs"].Engine(s, blob, max_batch=1, max_k=4, kv_capacity=ctx + 64)
    q = env["oracle"].Model(s, blob, table, ctx + 64).new_seq()
    env["harness"].inject_context(eng, q, s, 0, ctx, 5)
    p = hi.make_prompt(s.V, 16, seq=41)
    eng.prefill([p])
    q.prefill(p)
    want = np.asarray(q.conv()[1], np.float64)
    got = eng.export_state(1, 0, env["hs"].STATE_CONV).astype(np.float64)
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    print("error %.2e" % err)
    assert err < 5e-6 and eng.device_status() == 0


@pytest.mark.parametrize("name,n,max_k", [
    ("d512", 200, 4),        # down-projection K = 12288: 256 x 48 tiles in 12 segments, residual epilogue
    ("d1280", 1900, 4),      # out- and down-projection 256 x 144 tiles, both planes in one accumulator, residual epilogue
    ("d1024", 700, 8)])      # in-projection 256 x 240 tiles; residual projections 256 x 48, two accumulators
def test_wide_projection_forms(env, name, n, max_k):
    base = hi.CONFIGS["cfg1_tiny"].replace(V=512)
    s = {"d512": base.replace(d=512, ff=12288), "d1280": base.replace(d=1280, H=40, ff=2560, N=128),
         "d1024": hi.CONFIGS["cfg2_0p5b"].replace(L=2, V=512, ff=4096)}[name]
    blob, table = hi.make_weights(s, 0, "jitter")
    eng = env["hs"].Engine(s, blob, max_batch=1, max_k=max_k, kv_capacity=n + 16)
    model = env["oracle"].Model(s, blob, table, n + 16)
    p = hi.make_prompt(s.V, n, seq=7)
    q = model.new_seq()
    q.prefill(p)
    eng.prefill([p])
    env["harness"].compare_states(eng, [q], s, kv_rows=None)
    # logits of the last position: what the last layer's residual projections left
    T = max_k + 1
    row = (n - 1) % T
    q2 = model.new_seq()
    q2.prefill(p[:n - 1])
    want = q2.round(0, cand_in=np.asarray(p[n - 1:], np.int32), forced_n=0, want_logits=True)["logits"][0]
    got = eng.get_logits(row + 1)[row]
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    print(name, "logits %.2e" % err)
    assert err < 1e-4 and eng.device_status() == 0


@pytest.mark.parametrize("name", ["par64", "seq"])
def test_two_tokens_at_max_k_0(env, name):
    # two one-row passes: as many launches as two prompts of one token, and what the oracle has
    s = SHAPES[name]
    blob, table = hi.make_weights(s, 0, "jitter")
    eng = env["hs"].Engine(s, blob, max_batch=1, max_k=0, kv_capacity=16)
    model = env["oracle"].Model(s, blob, table, 16)
    p = hi.make_prompt(s.V, 2, seq=3)
    at = [eng.launch_count()]
    for prompt in ([p], [p[:1]]):
        eng.reset()
        eng.prefill(prompt)
        at.append(eng.launch_count())
    assert at[1] - at[0] == 2 * (at[2] - at[1])
    eng.reset()
    eng.prefill([p])
    q = model.new_seq()
    q.prefill(p)
    env["harness"].compare_states(eng, [q], s)
    assert eng.device_status() == 0
