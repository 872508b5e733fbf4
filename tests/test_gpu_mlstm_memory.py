"""mLSTM prompt scores where the memory for the states between segments cannot be had: the prompt
is taken chunk after chunk in what the features alone need."""
import numpy as np
import pytest
import torch

from workload import gen, get_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["q4b", "tiny"])
def test_prompt_without_segment_states(cuda_device, name):
    from paper_2607_05061_gb300 import kvpop
    cfg = get_config(name, batch=3)
    lengths = [449, 64, 1]
    H, G, d, D, P = cfg.n_kv_heads, cfg.q_per_kv, cfg.head_dim, cfg.delay_D, max(lengths)
    w = gen.mlstm_weights(cfg)
    K = gen.kv_tokens(cfg, "k", 0, 3, 0, P, device=cuda_device)
    V = gen.kv_tokens(cfg, "v", 0, 3, 0, P, device=cuda_device)
    Q = torch.zeros((3, H * G, P, d), dtype=K.dtype, device=cuda_device)
    caches = []
    try:
        for fail in (0, 1):
            cache = kvpop.KVpopCache(3, H, G, d, P, D, 4, cfg.kv_dtype, mlstm=w)
            kvpop.kvpop_debug_fail_alloc_after(fail)
            cache.prefill(Q, K, V, lengths)
            cache.check()
            caches.append(cache)
    finally:
        kvpop.kvpop_debug_fail_alloc_after(0)
    for b in range(3):
        for h in range(H):
            (pos, want), (pos2, got) = (c.pair_state(b, h) for c in caches)
            assert pos == pos2
            want, got = np.asarray(want), np.asarray(got)
            # the score bound of the parity tests, once for either form
            assert got.size == 0 or np.max(np.abs(got - want) / (1.0 + np.abs(want))) <= 2e-4
    for c in caches:
        c.free()
