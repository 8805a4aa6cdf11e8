"""Which attention kernel runs must not depend on what the process did before: each test here is the first thing that a process
of its own does with the library (needs a B200)."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _in_fresh_process(code):
    path = os.pathsep.join([ROOT, os.path.join(ROOT, "tests")])
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=ROOT, env=dict(os.environ, PYTHONPATH=path), timeout=300,
                       stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    assert r.returncode == 0, r.stdout[-3000:]


def test_allocation_free_attention_in_clusters_before_any_cache():
    _in_fresh_process("""
        import numpy as np, torch
        import paper_2608_22704_b200 as wnw
        from helpers import bf16_bits_to_f64, dense_attention
        from workloads.synth import bf16_bits
        n_q, n_kv, d, n = 8, 4, 64, 777
        gen = torch.Generator().manual_seed(5)
        kv = torch.full((n_kv, 2, 784, d), float("nan"), dtype=torch.bfloat16)
        kv[:, :, :n] = torch.randn(n_kv, 2, n, d, generator=gen).to(torch.bfloat16)
        q = (torch.randn(n_q, d, generator=gen) * 1.5).to(torch.bfloat16)
        kv_dev, q_dev = kv.cuda(), q.cuda()

        def attend():
            out = torch.full((n_q, d), float("nan"), dtype=torch.bfloat16, device="cuda")
            wnw.wnw_attend_static(kv_dev, n, q_dev, out)
            assert not wnw.wnw_attend_static_status()
            return out.cpu()

        first = attend()
        assert wnw.wnw_debug_attend_static_cluster(n, n_q, n_kv, d) == 4      # 49 granules: four pieces of at most 16
        assert wnw.wnw_debug_attend_static_cluster(128, n_q, n_kv, d) == 0    # one piece
        K, V, Q = (bf16_bits_to_f64(bf16_bits(x.contiguous())) for x in (kv[:, 0, :n], kv[:, 1, :n], q))
        want = np.stack([dense_attention(Q[h], K[h // 2], V[h // 2], 1.0 / np.sqrt(d))[0] for h in range(n_q)])
        assert np.abs(first.float().numpy() - want).max() <= 2e-2             # bf16 weights and outputs of O(1)
        wnw.wnw_destroy(wnw.wnw_create(1, n_q, n_kv, d, 1, 1024, 16, 16, 0.25, np.array([0, 1, 1, 2], np.uint8)))
        assert torch.equal(first, attend())                                   # the same kernel before and after a cache was made
    """)


# an anchor of one sequence: one CTA to an SM; of five (five clusters of 16 pieces): two to an SM
@pytest.mark.parametrize("audio,d,cut", [((2000,), 128, "SHORT"), ((3000,) * 5, 128, "SHORT_DENSE"), ((1500,), 64, "SHORT")])
def test_short_pieces_of_a_token_base_before_any_other_cache(audio, d, cut):
    _in_fresh_process(f"""
        import numpy as np
        import paper_2608_22704_b200 as wnw
        from parity_harness import Lockstep
        from workloads import ROLE_ANCHOR as A, ROLE_FIXED as F, ROLE_TIDAL as T, tiny_custom
        w = tiny_custom(n_layers=3, n_q_heads=8, n_kv_heads=2, head_dim={d}, n_text=7, audio_lens={audio}, chunk=25, budget=0.2, n_steps=5,
                        roles=[[A, T], [A, F], [T, A]], region=25, jump_every=2)
        ls = Lockstep(w, seed=61, oracle_seqs=[0], residency=wnw.WNW_RESIDENCY_SEGMENT_LAG_TOKEN_BASE, evict_lag=1, token_seg=25,
                      token_retention=np.full((3, 2), 0.2, np.float32))
        wnw.wnw_set_layer_dependency(ls.h, wnw.WNW_LAYERS_CHAINED)
        ls.prefill()
        for t in range(5):
            ls.decode_step(t, graph=t >= 2)
        cuts = [wnw.wnw_debug_get_layer_cut(ls.h, l) for l in range(3)]
        assert [c[0] for c in cuts] == [wnw.WNW_DEBUG_CUT_{cut}] * 3, cuts
        assert ls.max_out_err <= 2e-2
        ls.close()
    """)


def test_first_allocation_free_call_inside_a_capture():
    _in_fresh_process("""
        import torch
        import paper_2608_22704_b200 as wnw
        gen = torch.Generator().manual_seed(7)
        kv = torch.randn(4, 2, 784, 64, generator=gen).to(torch.bfloat16).cuda()
        q = torch.randn(8, 64, generator=gen).to(torch.bfloat16).cuda()
        outs = [torch.zeros_like(q) for _ in range(2)]
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            wnw.wnw_attend_static(kv, 777, q, outs[0], stream=stream)
        graph.replay()
        torch.cuda.synchronize()
        wnw.wnw_attend_static(kv, 777, q, outs[1])
        assert wnw.wnw_debug_attend_static_cluster(777, 8, 4, 64) == 4
        assert not wnw.wnw_attend_static_status()
        assert torch.equal(*outs) and outs[0].abs().max() > 0
    """)
