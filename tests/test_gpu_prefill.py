"""bf16 prompt passes on the prefill kernel (128 token rows x 256 features
per tile, activations as bf16 hi + lo pairs on the MMA's M side).

* The K/V cache a prefill writes, layer by layer, against the oracle's
  (float64 on the bf16-rounded weights, K/V rounded to bf16 as cached):
  every row of every layer within two bf16 steps of the largest entry, and
  the first generated token equal to the oracle's wherever its top-2 gap is
  clear.  Prompts are ragged (several 128-row tiles and a partial one); the
  shapes cover head_dim 64 and 128, GQA, a gate/up tail tile (d_ffn 688 is
  not a multiple of 128) and a K tail (688 is not a multiple of 64).
* A row's result does not depend on the pass it sits in: chunk sizes 16,
  128, 992 and the default (1024) write bit-identical caches.
"""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import OracleModel
from oracle.decode import prefill as oracle_prefill
from workloads import workload, make_weights, make_prompts
from gpu_helpers import rounded_weights

pytestmark = pytest.mark.gpu


def _case(name):
    if name == "tiny":
        return workload("tiny").with_(dtype="bf16", prompt_len=(300, 300))
    w = workload("1b")      # GQA 16/8, head_dim 128, d 2048, F 5632, two layers
    return w.with_(shape=replace(w.shape, n_layers=2), split_k=1, prompt_len=(700, 700))


def _prefill(w, dw, P, chunk):
    from paper_2510_05421_gb300 import DVIEngine
    eng = DVIEngine(w.shape, "bf16", dw, batch=1, k_spec=w.k_spec, split_k=w.split_k, lora_rank=w.lora_rank,
                    lora_gamma=w.lora_gamma, max_seq_len=len(P[0]) + 64, log_steps=w.update_every,
                    prefill_chunk=chunk)
    eng.prefill(0, torch.from_numpy(P[0]).cuda())
    st = eng.stats()
    s = w.shape
    shape = (s.n_layers, 1, s.n_kv_heads, len(P[0]) + 64, s.head_dim)
    k = eng.buffer("K_CACHE", torch.bfloat16).view(shape)[:, 0, :, :len(P[0])].float().cpu().numpy()
    v = eng.buffer("V_CACHE", torch.bfloat16).view(shape)[:, 0, :, :len(P[0])].float().cpu().numpy()
    first = int(eng.first[0].item())
    eng.close()
    assert st["device_status"] == 0, st["device_flags"]
    return k, v, first


@pytest.mark.parametrize("name", ["tiny", "1b-L2"])
def test_prefill_cache_matches_oracle(name):
    from paper_2510_05421_gb300 import DeviceWeights
    w = _case(name.split("-")[0])
    W = make_weights(w)
    P = make_prompts(w)
    n = len(P[0])
    k, v, first = _prefill(w, DeviceWeights.from_host(W, "bf16"), P, 0)
    m = OracleModel(rounded_weights(W), w.shape, w.lora_gamma, dtype=np.float64, kv_dtype="bf16")
    cache = m.new_cache(n + 1)
    tok, logits = oracle_prefill(m, cache, P[0])
    for l in range(w.shape.n_layers):
        for got, ref in ((k[l], cache.k[l, :n]), (v[l], cache.v[l, :n])):
            ref = ref.transpose(1, 0, 2)                 # [H_kv, n, hd] as the GPU stores it
            err = np.abs(got - ref).max() / np.abs(ref).max()
            assert err < 2 ** -7, (l, err)
    top2 = np.partition(logits, -2)[-2:]
    if top2[1] - top2[0] > 0.06:
        assert first == tok


def test_prefill_chunk_size_does_not_change_the_cache():
    from paper_2510_05421_gb300 import DeviceWeights
    w = _case("tiny")
    W = make_weights(w)
    P = make_prompts(w)
    dw = DeviceWeights.from_host(W, "bf16")
    outs = [_prefill(w, dw, P, c) for c in (16, 128, 992, 0)]
    for k, v, first in outs[1:]:
        assert np.array_equal(k, outs[0][0])
        assert np.array_equal(v, outs[0][1])
        assert first == outs[0][2]


# (query heads, KV heads, head_dim, prompt): one partial tile of 128 query
# vectors, tile and chunk edges, GQA groups that do not divide 128, and enough
# (row, head) pairs that a CTA takes two tiles
TILES = [(4, 4, 64, 1), (4, 4, 64, 127), (4, 4, 64, 129), (6, 2, 64, 130), (16, 2, 64, 257), (4, 2, 128, 128),
         (32, 32, 64, 700), (20, 20, 128, 1025)]


@pytest.mark.parametrize("hq,hkv,hd,n", TILES)
def test_attention_tiles(hq, hkv, hd, n):
    """Layer 2's K/V rows, which carry layer 1's attention output, against the
    oracle within two bf16 steps of the largest entry (2^-7 relative), and
    bit-identical whichever rows share a pass (chunks of 48 rows)."""
    from paper_2510_05421_gb300 import DeviceWeights
    from workloads import tiny_shape
    w = workload("tiny").with_(dtype="bf16", prompt_len=(n, n), split_k=1,
                               shape=tiny_shape(n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd))
    W = make_weights(w)
    P = make_prompts(w)
    dw = DeviceWeights.from_host(W, "bf16")
    k, v, first = _prefill(w, dw, P, 0)
    m = OracleModel(rounded_weights(W), w.shape, w.lora_gamma, dtype=np.float64, kv_dtype="bf16")
    cache = m.new_cache(n + 1)
    oracle_prefill(m, cache, P[0])
    for got, ref in ((k, cache.k), (v, cache.v)):
        for l in range(2):
            r = ref[l, :n].transpose(1, 0, 2)
            assert np.abs(got[l] - r).max() <= 2.0 ** -7 * np.abs(r).max(), l
    k2, v2, first2 = _prefill(w, dw, P, 48)
    assert np.array_equal(k, k2) and np.array_equal(v, v2) and first == first2


# (d, query heads, KV heads, head_dim, d_ffn, prompt): the 1B width at 1, 2, 3
# and 6 row tiles (QKV split 8, 4, 2 and 1 ways over K; O 8, 8, 4, 2; gate/up
# 2, 1; down 8, 8, 4, 2), a width with head_dim 64, and a d_ffn whose last K
# range is empty (33 K blocks over 8 ranges) and whose last tile is partial
SPLITS = [(2048, 16, 8, 128, 5632, 17), (2048, 16, 8, 128, 5632, 129), (2048, 16, 8, 128, 5632, 300),
          (2048, 16, 8, 128, 5632, 700), (1024, 16, 4, 64, 2816, 40), (1024, 8, 8, 128, 2088, 130)]


@pytest.mark.parametrize("d,hq,hkv,hd,f,n", SPLITS)
def test_short_prompts_split_over_k(d, hq, hkv, hd, f, n):
    """Prompts whose projections split K over a cluster: the caches against the
    oracle (as above) and bit-identical in passes of 48 rows."""
    from paper_2510_05421_gb300 import DeviceWeights
    from workloads import tiny_shape
    w = workload("tiny").with_(dtype="bf16", prompt_len=(n, n), split_k=1,
                               shape=tiny_shape(n_layers=2, d_model=d, n_heads=hq, n_kv_heads=hkv, head_dim=hd, d_ffn=f))
    W = make_weights(w)
    P = make_prompts(w)
    dw = DeviceWeights.from_host(W, "bf16")
    k, v, first = _prefill(w, dw, P, 0)
    m = OracleModel(rounded_weights(W), w.shape, w.lora_gamma, dtype=np.float64, kv_dtype="bf16")
    cache = m.new_cache(n + 1)
    oracle_prefill(m, cache, P[0])
    for got, ref in ((k, cache.k), (v, cache.v)):
        for l in range(2):
            r = ref[l, :n].transpose(1, 0, 2)
            assert np.abs(got[l] - r).max() <= 2.0 ** -7 * np.abs(r).max(), l
    k2, v2, first2 = _prefill(w, dw, P, 48)
    assert np.array_equal(k, k2) and np.array_equal(v, v2) and first == first2


# (query heads, KV heads, head_dim, prompt): the last chunk of 128 positions
# nearly empty and nearly full, two tiles of a CTA that end in different chunks,
# a full last chunk
STALE = [(4, 4, 64, 1), (4, 2, 128, 127), (16, 2, 64, 130), (32, 32, 64, 700), (20, 20, 128, 1025), (4, 4, 64, 256)]


@pytest.mark.parametrize("hq,hkv,hd,n", STALE)
def test_values_behind_the_prompt_do_not_matter(hq, hkv, hd, n):
    """A cache whose other rows (an earlier request's, the neighbouring heads'
    and sequences') are NaN: the prompt's K/V rows and first token are bit for
    bit those of a clean cache."""
    from paper_2510_05421_gb300 import DVIEngine, DeviceWeights
    from workloads import tiny_shape
    w = workload("tiny").with_(dtype="bf16", prompt_len=(n, n), split_k=1,
                               shape=tiny_shape(n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd))
    dw = DeviceWeights.from_host(make_weights(w), "bf16")
    prompt = torch.from_numpy(make_prompts(w)[0]).cuda()
    room = n + 9
    outs = []
    for stale in (0.0, float("nan")):
        eng = DVIEngine(w.shape, "bf16", dw, batch=2, k_spec=w.k_spec, split_k=1, lora_rank=w.lora_rank,
                        lora_gamma=w.lora_gamma, max_seq_len=room, log_steps=1)
        rows = [eng.buffer(b, torch.bfloat16) for b in ("K_CACHE", "V_CACHE")]
        for r in rows:
            r.fill_(stale)
        torch.cuda.synchronize()
        eng.prefill(0, prompt)
        eng.sync()
        assert eng.stats()["device_status"] == 0
        outs.append([r.view(2, 2, hkv, room, hd)[:, 0, :, :n].clone() for r in rows] + [int(eng.first[0])])
        eng.close()
    assert all(torch.isfinite(t).all() for t in outs[1][:2])
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    assert outs[0][2] == outs[1][2]
