"""The mLSTM prompt scores where a prompt's chunks are cut into segments: prompt lengths at the
chunk edges and segments of several chunks, against the recurrence in fp64."""
import numpy as np
import pytest
import torch

from oracle.mlstm import MlstmParams, MlstmState
from workload import gen, get_config

pytestmark = pytest.mark.gpu


def scores(w, h, K, V, D):
    st = MlstmState(MlstmParams.for_head(w, h), K.shape[1])
    out = []
    for t in range(K.shape[0]):
        st.update(np.concatenate([K[t], V[t]]))
        if t >= D:
            out.append(st.score(np.concatenate([K[t - D], V[t - D]])))
    return np.asarray(out)


# relative score bound of the parity tests (fp32 arithmetic over the whole recurrence)
TOL = 1e-4


@pytest.mark.parametrize("name,batch,lengths", [
    ("tiny", 3, [64, 65, 193]), ("q4b", 3, [63, 128, 321]), ("q4b", 4, [1, 130, 16, 17]),
    # 160 sequences x 8 heads of up to 1025 tokens: more than 256 MB between chunks, so a
    # segment holds several
    ("q4b", 160, [1025, 700, 449] + [5] * 157)])
def test_scores_at_segment_edges(cuda_device, name, batch, lengths):
    from paper_2607_05061_gb300 import kvpop
    cfg = get_config(name, batch=batch)
    w = gen.mlstm_weights(cfg)
    H, G, d, D, P = cfg.n_kv_heads, cfg.q_per_kv, cfg.head_dim, cfg.delay_D, max(lengths)
    B = P + 1                                            # everything is kept, in order
    dt = gen.torch_dtype(cfg.kv_dtype)
    cache = kvpop.KVpopCache(batch, H, G, d, B, D, 4, cfg.kv_dtype, mlstm=w)
    K, V = torch.zeros((2, batch, H, P, d), dtype=dt, device=cuda_device)
    for i, n in enumerate(lengths):
        K[i, :, :n] = gen.kv_tokens(cfg, "k", i, 1, 0, n, device=cuda_device)[0]
        V[i, :, :n] = gen.kv_tokens(cfg, "v", i, 1, 0, n, device=cuda_device)[0]
    Q = torch.zeros((batch, H * G, P, d), dtype=dt, device=cuda_device)
    cache.prefill(Q, K, V, lengths)
    st = kvpop.parse_state(cache.export_state(), cache.cfg) if batch < 10 else None
    for b, h in ((0, 0), (1, H - 1), (2, 1 % H)):
        n = lengths[b]
        want = scores(w, h, K[b, h, :n].double().cpu().numpy(), V[b, h, :n].double().cpu().numpy(), D)
        pos, got = cache.pair_state(b, h)
        assert pos == list(range(max(0, n - D)))
        got = np.asarray(got, dtype=np.float64)
        assert got.shape == want.shape
        assert got.size == 0 or np.max(np.abs(got - want) / (1.0 + np.abs(want))) <= TOL
        if st is None:
            continue
        # the state that decode goes on from, up to its common scale
        ref = MlstmState(MlstmParams.for_head(w, h), d)
        for t in range(n):
            ref.update(np.concatenate([K[b, h, t].double().cpu().numpy(), V[b, h, t].double().cpu().numpy()]))
        i = b * H + h
        scale = np.exp(float(st["mlstm_m"][i]) - ref.m)
        assert np.max(np.abs(st["mlstm_C"][i] * scale - ref.C)) <= TOL * np.max(np.abs(ref.C))
        assert np.max(np.abs(st["mlstm_z"][i] * scale - ref.z)) <= TOL * np.max(np.abs(ref.z))
    cache.free()
