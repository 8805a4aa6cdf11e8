"""The attention, scoring, token-compression and recall kernels at the sizes where their cuts change: edges of granules, tiles,
pieces and clusters, groups with padding heads, more text queries than a launch takes (needs a B200)."""
import numpy as np
import pytest
import torch

import paper_2608_22704_b200 as wnw
from helpers import bf16_bits_to_f64, dense_attention
from workloads import ROLE_ANCHOR as A, ROLE_FIXED as F, ROLE_TIDAL as T, Synth, tiny_custom
from workloads.synth import bf16_bits

pytestmark = pytest.mark.gpu
CLUSTER, WIDE, DENSE = wnw.WNW_DEBUG_CUT_CLUSTER, wnw.WNW_DEBUG_CUT_SHORT, wnw.WNW_DEBUG_CUT_SHORT_DENSE


def _cuts(ls):
    """Per layer: the attention kernel, CTAs of a cluster, whether a head takes several clusters."""
    return [wnw.wnw_debug_get_layer_cut(ls.h, l) for l in range(ls.w.n_layers)]


# audio tokens: one granule; a head of one piece and one of two (256 keys a piece); 16 pieces; more than 16 pieces' worth
@pytest.mark.parametrize("n_q,n_kv,d,audio", [(2, 2, 64, (16, 17)), (6, 2, 128, (255, 256, 257)), (16, 2, 128, (500,)), (18, 2, 128, (270,)),
                                              (32, 2, 64, (4097, 31)), (14, 2, 128, (3900, 4200))])
@pytest.mark.parametrize("mode", [wnw.WNW_LAYERS_CHAINED, wnw.WNW_LAYERS_SERIAL])
def test_chained_layers_clustered_pieces(n_q, n_kv, d, audio, mode):
    from parity_harness import Lockstep
    w = tiny_custom(n_layers=3, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=d, n_text=14, audio_lens=audio, chunk=16, budget=0.25, n_steps=5,
                    roles=[[A, T], [T, F], [F, A]], region=16, jump_every=2)
    ls = Lockstep(w, seed=41)
    try:
        wnw.wnw_set_layer_dependency(ls.h, mode)
        ls.prefill()
        for t in range(5):          # the new token's row crosses into a second text granule (14 + 2)
            ls.decode_step(t, graph=t >= 2, check_slots=(t == 4))
        ls.check_stats()
        assert ls.max_out_err <= 2e-2
    finally:
        ls.close()


# Short pieces of one and of two CTAs to an SM: one piece and 16 of 16 granules exactly, one granule more (the cut of longer pieces),
# groups with padding heads, the new token's row in either half of a granule and across two; chunks that fill granules partly
@pytest.mark.parametrize("n_q,n_kv,d,chunk,audio,n_text,form", [
    (8, 2, 128, 16, (224,), 6, WIDE), (8, 2, 128, 16, (4064,), 14, WIDE), (8, 2, 128, 16, (4065,), 14, CLUSTER), (5, 5, 64, 16, (300,), 0, WIDE),
    (12, 4, 128, 16, (4000, 3900, 3000, 17), 6, DENSE), (8, 4, 64, 16, (4064, 4064, 4064, 60), 15, DENSE),
    (64, 4, 64, 25, (2500, 2500, 2500, 26), 13, DENSE), (10, 2, 128, 25, (1990,) * 8, 7, DENSE),
    (12, 4, 128, 16, (4000, 3900, 17), 6, None), (8, 4, 64, 16, (4064, 4064, 900, 60), 15, None),   # near the line between the two
    (64, 4, 64, 25, (1500, 2500, 1700, 26), 13, None),
    (64, 4, 128, 16, (2000,) * 4, 7, None)])   # 16 query heads a KV head of 128: one kernel for both
def test_chained_layers_of_short_pieces(n_q, n_kv, d, chunk, audio, n_text, form):
    from parity_harness import Lockstep
    roles = [[(A, T, F, T, A)[(h + l) % 5] for h in range(n_kv)] for l in range(3)]
    w = tiny_custom(n_layers=3, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=d, n_text=n_text, audio_lens=audio, chunk=chunk, budget=0.25, n_steps=6,
                    roles=roles, region=chunk, jump_every=2)
    ls = Lockstep(w, seed=53, oracle_seqs=[0, len(audio) - 1] if len(audio) > 1 else [0])
    try:
        wnw.wnw_set_layer_dependency(ls.h, wnw.WNW_LAYERS_CHAINED)
        ls.prefill()
        for t in range(6):
            ls.decode_step(t, graph=t >= 2)
        cuts = _cuts(ls)
        assert cuts[0][0] == form or form is None and cuts[0][0] in (WIDE, DENSE), cuts   # the first layer has an anchor of every sequence
        assert all(c[0] in (WIDE, DENSE) for c in cuts[1:]) and not any(c[2] for c in cuts), cuts
        assert ls.max_out_err <= 2e-2
    finally:
        ls.close()


# Heads of more than 384 granules take several clusters: one granule less (the cut of longer pieces) and more, five clusters, ten, a
# part of a batch; token bases
@pytest.mark.parametrize("n_q,n_kv,d,chunk,audio,n_text,residency,several", [
    (8, 2, 128, 16, (6112,), 6, 0, False), (8, 2, 128, 16, (6144, 40), 6, 0, True), (10, 2, 128, 64, (17000,), 14, 0, True),
    (32, 2, 128, 16, (6200,), 7, 0, True), (32, 2, 64, 16, (9000, 300, 6300), 3, 0, True), (8, 2, 64, 25, (5000,), 15, 2, True),
    (8, 2, 128, 25, (5300, 700), 7, 2, True), (8, 2, 64, 16, (40000,), 27, 0, True), (8, 2, 128, 16, (40000,), 27, 0, True)])
def test_chained_heads_of_several_clusters(n_q, n_kv, d, chunk, audio, n_text, residency, several):
    from parity_harness import Lockstep
    w = tiny_custom(n_layers=3, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=d, n_text=n_text, audio_lens=audio, chunk=chunk, budget=0.2, n_steps=5,
                    roles=[[A, T], [T, F], [F, A]], region=chunk, jump_every=2)
    extra = dict(residency=residency, evict_lag=1, token_retention=np.full((3, n_kv), 0.2, np.float32), token_seg=25) if residency else {}
    ls = Lockstep(w, seed=59, gen_device="cuda:0", **extra)
    try:
        wnw.wnw_set_layer_dependency(ls.h, wnw.WNW_LAYERS_CHAINED)
        ls.prefill(check_slots=False)
        for t in range(5):
            ls.decode_step(t, graph=t >= 2)
        cuts = _cuts(ls)
        for l in (0, 2):   # the layers with an anchor
            assert (cuts[l][0] in (WIDE, DENSE) and cuts[l][2]) if several else cuts[l] == (CLUSTER, 16, False), cuts
        assert ls.max_out_err <= 2e-2
    finally:
        ls.close()


# Longer pieces: 1408 granules, 3 of them text, are the longest head whose pieces share a cluster, in an e4m3 tier and where the
# short pieces of the long heads do not fit; alone they take several clusters.  Layers without a long head stay clustered
@pytest.mark.parametrize("audio,d,fp8,cut", [
    ((22480,), 128, True, "cluster"), ((22481,), 128, True, "none"), ((22600, 500), 128, True, "none"), ((40000,), 128, True, "none"),
    ((22480,) * 3, 64, False, "cluster"), ((22481, 22000, 22000), 64, False, "none"), ((22481,) * 3, 128, False, "none"),
    ((22480,), 64, False, "several"), ((22481,), 64, False, "several"), ((22600, 500), 128, False, "several"), ((40000,), 128, False, "several")])
def test_chained_layers_around_the_longest_clustered_head(audio, d, fp8, cut):
    from parity_harness import Lockstep
    w = tiny_custom(n_layers=4, n_q_heads=8, n_kv_heads=2, head_dim=d, n_text=27, audio_lens=audio, chunk=16, budget=0.1, n_steps=6,
                    roles=[[A, T], [T, F], [T, A], [T, T]], region=16, jump_every=2)
    ls = Lockstep(w, seed=47, gen_device="cuda:0", oracle_seqs=None if len(audio) < 3 else [0], kv_fp8=fp8)
    try:
        wnw.wnw_set_layer_dependency(ls.h, wnw.WNW_LAYERS_CHAINED)
        ls.prefill(check_slots=False)
        for t in range(6):
            ls.decode_step(t, graph=t >= 2, check_slots=(t == 5))
        ls.check_stats()
        cuts = _cuts(ls)
        for l in (0, 2):   # the layers with an anchor
            assert cuts[l] == (CLUSTER, 16, False) if cut == "cluster" else cuts[l][1] == 0 if cut == "none" else cuts[l][2], cuts
        assert all(cuts[l][1] > 0 for l in (1, 3)), cuts
        assert ls.max_out_err <= 2e-2
    finally:
        ls.close()


@pytest.mark.parametrize("n_q,n_kv,d", [(8, 4, 64), (16, 1, 128), (9, 3, 128), (128, 64, 64)])
def test_static_attention_edges(n_q, n_kv, d):
    dev = torch.device("cuda:0")
    gen = torch.Generator(device="cpu").manual_seed(n_q + d)
    for n in (1, 15, 16, 17, 127, 128, 129, 2400, 2401):
        padded = (n + 15) // 16 * 16
        kv = torch.randn(n_kv, 2, padded, d, generator=gen).to(torch.bfloat16).to(dev)
        q = (torch.randn(n_q, d, generator=gen) * 1.5).to(torch.bfloat16).to(dev)
        out = torch.full((n_q, d), float("nan"), dtype=torch.bfloat16, device=dev)
        wnw.wnw_attend_static(kv, n, q, out)
        K, V, Q = (bf16_bits_to_f64(bf16_bits(x.cpu().contiguous())) for x in (kv[:, 0, :n], kv[:, 1, :n], q))
        want = np.stack([dense_attention(Q[h], K[h * n_kv // n_q], V[h * n_kv // n_q], 1.0 / np.sqrt(d))[0] for h in range(n_q)])
        assert np.abs(out.float().cpu().numpy() - want).max() <= 2e-2, n
    assert not wnw.wnw_attend_static_status()


# a cluster a head: 2, 4, 5, 8, 9 and 16 pieces of 16 granules and one granule more; rows behind the clip hold NaN
@pytest.mark.parametrize("n_q,n_kv,d", [(8, 4, 64), (3, 1, 128), (32, 2, 128), (48, 3, 64)])
def test_static_attention_in_clusters(n_q, n_kv, d):
    dev = torch.device("cuda:0")
    gen = torch.Generator(device="cpu").manual_seed(n_q * d)
    for n in (130, 257, 1024, 1025, 2048, 2049, 4095, 4096, 4097):
        kv = torch.full((n_kv, 2, (n + 47) // 16 * 16, d), float("nan"), dtype=torch.bfloat16)
        kv[:, :, :n] = torch.randn(n_kv, 2, n, d, generator=gen).to(torch.bfloat16)
        q = (torch.randn(n_q, d, generator=gen) * 1.5).to(torch.bfloat16)
        out = torch.full((n_q, d), float("nan"), dtype=torch.bfloat16, device=dev)
        wnw.wnw_attend_static(kv.to(dev), n, q.to(dev), out)
        K, V, Q = (bf16_bits_to_f64(bf16_bits(x.contiguous())) for x in (kv[:, 0, :n], kv[:, 1, :n], q))
        want = np.stack([dense_attention(Q[h], K[h * n_kv // n_q], V[h * n_kv // n_q], 1.0 / np.sqrt(d))[0] for h in range(n_q)])
        assert np.abs(out.float().cpu().numpy() - want).max() <= 2e-2, n   # bf16 weights and outputs of O(1)
        pieces = -(-n // 256)
        assert wnw.wnw_debug_attend_static_cluster(n, n_q, n_kv, d) == (4 if pieces <= 4 else 8 if pieces <= 8 else 16 if pieces <= 16 else 0)
    assert not wnw.wnw_attend_static_status()


@pytest.mark.parametrize("n_queries", [8, 9, 17])
def test_scoring_takes_several_queries_per_launch(n_queries):
    from parity_harness import Lockstep
    w = tiny_custom(n_layers=2, n_q_heads=6, n_kv_heads=3, head_dim=128, n_text=3, audio_lens=(127, 400), chunk=25, budget=0.3, n_steps=2,
                    roles=[[A, T, F], [F, T, T]], region=25)
    w.n_prefill_queries = n_queries
    ls = Lockstep(w, seed=42)
    try:
        ls.prefill()                # scores, sets, tables and slots against the oracle
        ls.decode_step(0, check_slots=True)
        ls.decode_step(1, check_slots=True)
        ls.check_stats()
    finally:
        ls.close()


# tiles of 128 positions, 16 query rows a pass: one, two and three passes
@pytest.mark.parametrize("n_queries,audio", [(1, (123, 124)), (8, (125, 252)), (9, (1024,)), (20, (300,))])
def test_token_scores_over_tiles_and_passes(n_queries, audio):
    from parity_harness import Lockstep
    w = tiny_custom(n_layers=2, n_q_heads=8, n_kv_heads=4, head_dim=64, n_text=4, audio_lens=audio, chunk=32, budget=0.5, n_steps=2,
                    roles=[[A, T, F, F], [T, F, T, F]], region=32)
    w.n_prefill_queries = n_queries
    ret = np.array([[1.0, 1.0, 0.4, 0.25], [1.0, 0.3, 1.0, 0.5]], np.float32)
    ls = Lockstep(w, seed=43, token_retention=ret, token_seg=25)
    try:
        ls.prefill()                # per-position scores and kept positions against the oracle
        ls.decode_step(0)
        ls.decode_step(1)
        assert ls.max_out_err <= 2e-2
    finally:
        ls.close()


@pytest.mark.parametrize("chunk,n_kv,batch", [(1, 2, 1), (25, 3, 3), (33, 4, 40)])
def test_recall_moves_chunks_without_their_padding(chunk, n_kv, batch):
    """Chunks that fill their granules partly, many sequences (more than a warp looks up at once): slots stay bit-exact."""
    from parity_harness import Lockstep
    w = tiny_custom(n_layers=2, n_q_heads=n_kv, n_kv_heads=n_kv, head_dim=64, n_text=3, audio_lens=(6 * chunk + chunk // 2 + 1,) * batch, chunk=chunk,
                    budget=0.5, n_steps=4, roles=[[A] + [T] * (n_kv - 1), [T] * n_kv], region=max(chunk, 2), jump_every=1)
    ls = Lockstep(w, seed=44, oracle_seqs=[0, batch - 1] if batch > 1 else [0])
    try:
        ls.prefill()
        for t in range(4):
            ls.decode_step(t, graph=t >= 2, check_slots=True)
        assert ls.max_out_err <= 2e-2
    finally:
        ls.close()


def test_appends_queue_behind_steps_without_a_wait():
    """Audio arriving between eager and replayed steps with nothing drained: the outputs of the drained run."""
    w = tiny_custom(n_layers=3, n_q_heads=4, n_kv_heads=2, head_dim=64, n_text=4, audio_lens=(200,), chunk=16, budget=0.25, n_steps=8,
                    roles=[[A, T], [T, T], [A, T]], region=16, jump_every=2)
    syn, dev = Synth(w, seed=45, device="cuda:0"), torch.device("cuda:0")
    dec = [syn.decode(0, l) for l in range(3)]
    extra = torch.randn(2, 3, 4, 10, 2, 64, generator=torch.Generator(device=dev).manual_seed(5), device=dev).to(torch.bfloat16)

    def run(drained):
        h = wnw.wnw_create(3, 4, 2, 64, 1, 240, w.text_capacity, 16, 0.25, w.roles, streaming_audio=1)
        try:
            st = torch.cuda.Stream()
            for l in range(3):
                p = syn.prefill(0, l)
                wnw.wnw_place_prefill(h, 0, l, p["k"], p["v"], p["audio_begin"], p["audio_end"], p["q_last"])
                torch.cuda.synchronize()
            outs = []
            with torch.cuda.stream(st):
                for t in range(8):
                    if t % 2 == 0:
                        for l in range(3):
                            wnw.wnw_append_audio(h, 0, l, extra[0, l, t // 2], extra[1, l, t // 2], stream=st)
                    out = torch.zeros(3, 1, 4, 64, dtype=torch.bfloat16, device=dev)
                    wnw.wnw_step_begin(h, [0])
                    for l in range(3):
                        wnw.wnw_decode_layer(h, l, dec[l]["q"][t:t + 1], dec[l]["k_new"][t:t + 1], dec[l]["v_new"][t:t + 1], out[l], stream=st)
                    wnw.wnw_step_end(h, stream=st)
                    outs.append(out)
                    if drained:
                        wnw.wnw_sync(h)
            wnw.wnw_sync(h)
            return outs, [wnw.wnw_get_residency(h, 0, l) for l in range(3)]
        finally:
            wnw.wnw_destroy(h)

    a, b = run(True), run(False)
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x, y)
    for (t1, s1), (t2, s2) in zip(a[1], b[1]):
        assert np.array_equal(t1, t2) and np.array_equal(s1, s2)
