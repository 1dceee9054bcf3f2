"""Decode calls that leave most SMs idle run as clusters of four CTAs per 2048-key chunk where the head size is 128
and contexts are long (tik_decode_cluster.cu).  Rows and log-sum-exps equal those of the packed train-forward bit for bit: group
sizes, head sizes, page sizes, tile counts from one to sixteen (fewer tiles than CTAs among them), chunk
boundaries, and keys that grow along the sequence, so that the reference maximum moves and O is rescaled."""
import numpy as np
import pytest
import torch

from paper_2609_35140_b200 import synth
from gpu_common import count_diff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tik():
    from paper_2609_35140_b200 import binding
    binding.load()
    yield binding
    assert binding.device_status() == 0


@pytest.mark.parametrize("lens,Hkv,G,d,page,ramp", [
    ([1], 1, 1, 128, 64, 0.0), ([128, 129], 1, 8, 128, 16, 0.0), ([300, 511, 640], 2, 7, 128, 64, 0.0),
    ([2048], 4, 7, 128, 64, 3.0), ([2047, 1500, 77], 8, 8, 128, 128, 3.0),
    ([4321], 4, 7, 128, 64, 1.0), ([2049, 4096, 4097], 4, 4, 128, 32, 2.0),             # several chunks: partials
    ([1000] * 12, 5, 3, 128, 16, 3.0), ([2000, 30, 129, 257, 2048] * 3, 4, 8, 128, 64, 2.0),
    ([160], 1, 4, 64, 16, 0.0), ([2048, 100, 900], 8, 8, 64, 64, 3.0), ([5000, 3000], 6, 5, 64, 128, 2.0)])
def test_cluster_decode_equals_train_rows(tik, lens, Hkv, G, d, page, ramp):
    S = len(lens)
    w = synth.custom_workload([1] * S, [L - 1 for L in lens], G * Hkv, Hkv, d, page, index=70)
    q, k, v, cu = synth.make_qkv(w, "cuda")
    cu_h = w.cu_seqlens()
    for s in range(S):
        pos = torch.arange(lens[s], device="cuda")
        k[int(cu_h[s]):int(cu_h[s + 1])] *= (1.0 + ramp * (pos // 128) / 8.0).to(k.dtype)[:, None, None]
    lse_train = torch.zeros(q.shape[0], w.Hq, dtype=torch.float32, device="cuda")
    o_train = tik.tik_attn_train_fwd(q, k, v, cu, max(lens), w.softmax_scale, lse=lse_train)
    layout = synth.make_paged_layout(w)
    bt = torch.from_numpy(layout.block_table).cuda()
    kc = torch.full((layout.num_pages, Hkv, page, d), 2.0, dtype=torch.bfloat16, device="cuda")   # stale finite values
    vc = torch.full_like(kc, -3.0)
    ctx = torch.tensor(lens, dtype=torch.int32, device="cuda")
    tik.tik_kv_cache_write(k, v, cu, ctx, kc, vc, bt)
    rows = torch.tensor([int(cu_h[s]) + L - 1 for s, L in enumerate(lens)], device="cuda")
    for repeat in range(3):
        o = torch.full((S, w.Hq, d), 7.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.zeros(S, w.Hq, dtype=torch.float32, device="cuda")
        tik.tik_attn_decode(q[rows].contiguous(), ctx, kc, vc, bt, max(lens), w.softmax_scale, o=o, lse=lse)
        assert count_diff(o, o_train[rows]) == 0
        assert count_diff(lse, lse_train[rows]) == 0
    # an empty slot is left alone, shorter contexts than the host's bound as they are
    ctx2 = torch.tensor([0] + [max(1, L // 2) for L in lens[1:]], dtype=torch.int32, device="cuda")
    rows2 = torch.tensor([int(cu_h[s]) + max(1, L // 2) - 1 for s, L in enumerate(lens)], device="cuda")
    o = torch.full((S, w.Hq, d), 7.0, dtype=torch.bfloat16, device="cuda")
    tik.tik_attn_decode(q[rows2].contiguous(), ctx2, kc, vc, bt, max(lens), w.softmax_scale, o=o)
    assert bool((o[0] == 7.0).all()) and count_diff(o[1:], o_train[rows2][1:]) == 0


@pytest.mark.parametrize("S,Hkv,G,lo,hi", [(3, 2, 4, 1, 128), (3, 2, 4, 100, 129), (37, 4, 2, 1500, 2048), (38, 4, 2, 1500, 2048),
                                           (150, 8, 1, 4097, 4300)])
def test_decode_at_the_edges_of_the_kernel_choice(tik, S, Hkv, G, lo, hi):
    """Contexts of one tile and one key more, as many chunks as SMs and a few more, and many pairs of three
    chunks: the rows equal those of the packed train-forward."""
    rng = np.random.default_rng(S + hi)
    lens = [hi] + [int(x) for x in rng.integers(lo, hi + 1, S - 1)]
    w = synth.custom_workload([1] * S, [L - 1 for L in lens], G * Hkv, Hkv, 128, 64, index=71)
    q, k, v, cu = synth.make_qkv(w, "cuda")
    o_train = tik.tik_attn_train_fwd(q, k, v, cu, hi, w.softmax_scale)
    layout = synth.make_paged_layout(w)
    kc, vc = synth.fill_paged_cache(w, layout, k, v)
    ctx = torch.tensor(lens, dtype=torch.int32, device="cuda")
    rows = torch.tensor([int(w.cu_seqlens()[s]) + L - 1 for s, L in enumerate(lens)], device="cuda")
    o = tik.tik_attn_decode(q[rows].contiguous(), ctx, kc, vc, torch.from_numpy(layout.block_table).cuda(), hi, w.softmax_scale)
    assert count_diff(o, o_train[rows]) == 0


@pytest.mark.parametrize("chunks,Hkv,G,page", [(32, 4, 7, 64), (33, 3, 8, 16), (34, 2, 4, 64), (37, 1, 8, 32), (38, 2, 1, 128)])
def test_cluster_decode_up_to_the_clusters_that_fit(tik, chunks, Hkv, G, page):
    """Calls of as many chunks as clusters fit on the device, of a few more and a few less, most contexts a tile or
    two long under a bound of one chunk: the rows equal those of the packed train-forward."""
    S = -(-chunks // Hkv)
    lens = ([2048] + 8 * [1, 127, 128, 129, 300, 511, 640, 1025])[:S]
    w = synth.custom_workload([1] * S, [L - 1 for L in lens], G * Hkv, Hkv, 128, page, index=72)
    q, k, v, cu = synth.make_qkv(w, "cuda")
    o_train = tik.tik_attn_train_fwd(q, k, v, cu, 2048, w.softmax_scale)
    layout = synth.make_paged_layout(w)
    kc, vc = synth.fill_paged_cache(w, layout, k, v)
    ctx = torch.tensor(lens, dtype=torch.int32, device="cuda")
    rows = torch.tensor([int(w.cu_seqlens()[s]) + L - 1 for s, L in enumerate(lens)], device="cuda")
    o = tik.tik_attn_decode(q[rows].contiguous(), ctx, kc, vc, torch.from_numpy(layout.block_table).cuda(), 2048, w.softmax_scale)
    assert count_diff(o, o_train[rows]) == 0
