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
