"""Speculative sampling at vocabularies where its split over eight CTAs can go wrong: shares that are empty, ragged, not a
multiple of four ids, more than one sweep per thread, and more than one group of 32 ids per block (against the CPU oracle, decision margins as in harness.py)."""
import numpy as np
import pytest

import hs_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,tau", [(31, 0.3), (257, 0.1), (1003, 0.05), (33001, 0.02), (262201, 0.01)])
def test_sampling_vocabulary_sizes(V, tau):
    import oracle
    from paper_2605_01106_b200 import build, binding as hs
    build.build()
    import harness
    s = hi.CONFIGS["cfg1_tiny"].replace(V=V)
    blob, table = hi.make_weights(s, 0, "jitter")
    eng = hs.Engine(s, blob, max_batch=2, max_k=4, kv_capacity=128)
    model = oracle.Model(s, blob, table, 128)
    prompts = [hi.make_prompt(s.V, n, seq=b) for b, n in enumerate((12, 7))]
    seqs = [model.new_seq() for _ in prompts]
    for q, p in zip(seqs, prompts):
        q.prefill(p)
    eng.prefill(prompts)
    rep, full = harness.run_rounds_sampled(eng, seqs, s, 4, 16, tau)
    print(V, tau, rep, "rounds compared in full:", full)
    # (how many rounds have wide decision margins is the oracle's matter: ten decisions a round)
    assert full >= 2 and eng.device_status() == 0
