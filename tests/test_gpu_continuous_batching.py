"""Sequences joining and leaving between steps: every step serves its own active set, a finished sequence's slot is
re-placed with a fresh prefill while the others keep decoding, and captured steps are re-captured when the set changes.
Everything in lock-step with the oracle (needs a B200)."""
import numpy as np
import pytest
import torch

import paper_2608_22704_b200 as wnw
from workloads import ROLE_ANCHOR, ROLE_FIXED, ROLE_TIDAL, config4, tiny_custom
from workloads.synth import bf16_bits

pytestmark = pytest.mark.gpu
A, T, F = ROLE_ANCHOR, ROLE_TIDAL, ROLE_FIXED


def _replace(ls, b):
    """Places sequence b's prefill again (a new request taking over the slot): state, tables and counters start over."""
    w = ls.w
    for l in range(w.n_layers):
        p = ls.syn.prefill(b, l)
        k, v, ql = (p[n].to(ls.dev) for n in ("k", "v", "q_last"))
        wnw.wnw_place_prefill(ls.h, b, l, k, v, p["audio_begin"], p["audio_end"], ql)
        ls.o.place_prefill(b, l, bf16_bits(p["k"]), bf16_bits(p["v"]), p["audio_begin"], p["audio_end"], bf16_bits(p["q_last"]))
    wnw.wnw_sync(ls.h)
    ls._steps[b] = 0
    for l in range(w.n_layers):
        if (w.roles[l] == T).any():
            g_tab, g_stamp = wnw.wnw_get_residency(ls.h, b, l)
            o_tab, o_stamp = ls.o.residency(b, l)
            assert g_tab.tolist() == o_tab.tolist() and g_stamp.tolist() == o_stamp.tolist()
    assert wnw.wnw_get_seq_dims(ls.h, b) == ls.o.dims(b)


@pytest.mark.parametrize("residency", [0, 1])
def test_sequences_join_leave_and_slots_are_reused(residency):
    from parity_harness import Lockstep
    roles = [[A, T, T, F], [T, F, T, F], [A, T, F, T]]
    w = tiny_custom(n_layers=3, n_q_heads=8, n_kv_heads=4, head_dim=64, n_text=6, audio_lens=(400, 170, 640, 90), chunk=25,
                    budget=0.2, n_steps=14, roles=roles, region=25, jump_every=3)
    ls = Lockstep(w, seed=21, residency=residency, evict_lag=2)
    try:
        ls.prefill()
        schedule = [[0, 1, 2, 3], [0, 1, 2, 3], [0, 2, 3], [0, 2], [2], [2, 1], [1, 2, 3], [3, 1, 2, 0], [0], [0, 1, 2, 3]]
        for t, act in enumerate(schedule):
            if t == 5:
                _replace(ls, 1)          # sequence 1 left after step 1; a new request takes its slot
            if t == 8:
                _replace(ls, 3)
            ls.decode_step(t, active=act, check_slots=True)
        # per-sequence step counts: what each slot decoded since its last placement
        assert ls._steps == {0: 7, 1: 4, 2: 9, 3: 1}
        for b in range(4):
            T_a, T_t, C, S = wnw.wnw_get_seq_dims(ls.h, b)
            assert T_t == w.n_text + ls._steps[b]
    finally:
        ls.close()


def test_graph_is_recaptured_when_the_active_set_changes():
    from parity_harness import Lockstep
    roles = [[A, T], [T, F]]
    w = tiny_custom(n_layers=2, n_q_heads=4, n_kv_heads=2, head_dim=64, n_text=4, audio_lens=(300, 200, 500), chunk=16,
                    budget=0.25, n_steps=10, roles=roles)
    ls = Lockstep(w, seed=5)
    try:
        ls.prefill()
        ls.decode_step(0, active=[0, 1, 2], graph=True, check_slots=True)
        ls.decode_step(1, active=[0, 1, 2], graph=True, check_slots=True)
        ls.decode_step(2, active=[0, 2], check_slots=True)            # eager step of another set: the work lists change
        with pytest.raises(wnw.WnwError):                             # the captured step is stale now: refused, not replayed
            wnw.wnw_graph_launch(ls.h, ls._gstream)
        for t, act in enumerate([[0, 2], [2, 1], [2, 1], [1], [1]], start=3):
            if t in (3, 4, 6):
                ls._graph = None                                      # capture again for the new set
            ls.decode_step(t, active=act, graph=True, check_slots=True)
    finally:
        ls.close()


def _split_recall_launches(w):
    """Recall launches of a replayed chained step that fills the machine: one inside the step for every layer of the first half
    whose tail updates tables, one behind the step for all the others."""
    L = w.n_layers
    anchor = [l for l in range(L) if (w.roles[l] == A).any()]
    tails = {max(l, min(anchor, key=lambda a: (abs(a - l), a))) for l in range(L) if (w.roles[l] == T).any()}
    half = (L + 1) // 2
    inside = sum(t < half for t in tails)
    assert 0 < inside < len(tails)
    return inside + 1


@pytest.mark.parametrize("dependency", [wnw.WNW_LAYERS_CHAINED, wnw.WNW_LAYERS_BATCHED])
def test_few_sequences_decode_on_after_steps_that_filled_the_machine(dependency):
    """Chained replays of twelve long sequences recall half of their layers inside the step and half behind it.  Most requests
    finish; the steps of the ones that are left are small, recall behind the step altogether, and their tidal heads wait for
    every layer's epoch: call by call, newly captured, and (all layers issued together) with the selection waiting too."""
    from parity_harness import Lockstep
    w = config4(budget=0.1, batch=12, n_steps=12)
    w.n_layers = 4; w.roles = w.roles[:4]; w.jump_every = 2
    ls = Lockstep(w, seed=17, gen_device="cuda:0", oracle_seqs=[0, 7])
    everyone, left = list(range(12)), [7]

    def steps(ts, active, graph):
        before = wnw.wnw_get_launch_counts(ls.h)[2]
        ls._graph = None
        for t in ts:
            ls.decode_step(t, active=active, graph=graph, check_slots=True)
        return wnw.wnw_get_launch_counts(ls.h)[2] - before

    try:
        wnw.wnw_set_layer_dependency(ls.h, wnw.WNW_LAYERS_CHAINED)
        ls.prefill(check_slots=False)
        assert steps([0, 1, 2], everyone, True) == 3 * _split_recall_launches(w)     # the form that the first half takes part in
        assert steps([3], left, False) == 1
        wnw.wnw_set_layer_dependency(ls.h, dependency)
        assert steps([4, 5], left, True) == 2
        assert steps([6], left, False) == 1
        wnw.wnw_set_layer_dependency(ls.h, wnw.WNW_LAYERS_CHAINED)
        assert steps([7, 8], everyone, True) == 2 * _split_recall_launches(w)
        wnw.wnw_set_layer_dependency(ls.h, dependency)
        assert steps([9, 10], left, True) == 2
    finally:
        ls.close()
