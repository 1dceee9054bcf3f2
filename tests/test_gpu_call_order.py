"""Calls queued back to back (every kernel may start under the tail of the one before) give the bits of
the same calls with a synchronisation after each: a layer whose every operator reads its predecessor's
output and whose buffers are written again by the next round."""
import pytest
import torch

from paper_2609_35140_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tik():
    from paper_2609_35140_b200 import binding
    binding.load()
    yield binding
    assert binding.device_status() == 0


@pytest.mark.parametrize("n", [3, 200])
def test_queued_calls_equal_synchronised_calls(tik, n):
    Hq, Hkv, d, H, inter, V, page, ctx_len = 8, 2, 128, 512, 704, 3000, 64, 300
    g = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *s, std=1.0: (torch.randn(*s, generator=g, device="cuda") * std).to(torch.bfloat16)
    blocks = -(-ctx_len // page)
    table = torch.randperm(n * blocks, generator=g, device="cuda").view(n, blocks).to(torch.int32)
    kc0, vc0 = rnd(n * blocks, Hkv, page, d), rnd(n * blocks, Hkv, page, d)
    ctx = torch.full((n,), ctx_len, dtype=torch.int32, device="cuda")
    cu = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    rope = synth.make_rope_table(ctx_len, d, device="cuda")
    w_q, w_k, w_v = rnd(Hq * d, H, std=0.05), rnd(Hkv * d, H, std=0.05), rnd(Hkv * d, H, std=0.05)
    w_o, w_gu, w_d, head = rnd(H, Hq * d, std=0.05), rnd(2 * inter, H, std=0.05), rnd(H, inter, std=0.05), rnd(V, H, std=0.05)
    norm, norm_d = rnd(H), rnd(d)
    ids = torch.randint(0, V, (n,), generator=g, device="cuda").to(torch.int32)
    x0 = rnd(n, H)

    def rounds(sync):
        step = torch.cuda.synchronize if sync else (lambda: None)
        kc, vc, x, out = kc0.clone(), vc0.clone(), x0.clone(), []
        h, y = torch.empty_like(x), torch.empty_like(x)      # written again by every round
        for _ in range(4):
            tik.tik_rmsnorm(x, norm, 1e-6, y=h); step()
            q, k, v = (tik.tik_linear(h, w).view(n, -1, d) for w in (w_q, w_k, w_v)); step()
            tik.tik_qk_norm_rope_kv_write(q, k, v, norm_d, norm_d, 1e-6, rope, cu, ctx, kc, vc, table); step()
            tik.tik_kv_cache_write(k, v, cu, ctx, kc, vc, table); step()
            o = tik.tik_attn_decode(q, ctx, kc, vc, table, ctx_len, 0.09); step()
            a = tik.tik_linear(o.view(n, -1), w_o); step()
            tik.tik_rmsnorm(a, norm, 1e-6, residual=x, y=h); step()
            m = tik.tik_swiglu(tik.tik_linear(h, w_gu)); step()
            tik.tik_linear(m, w_d, y=y); step()
            tik.tik_rmsnorm(y, norm, 1e-6, residual=x, y=h); step()
            out += [tik.tik_token_logprob(h, head, ids), x.clone()]; step()
        return out + [kc, vc]

    a, b = rounds(True), rounds(False)
    assert all(torch.equal(s, t) for s, t in zip(a, b))


@pytest.mark.parametrize("Hq,Hkv,d,lens", [(4, 1, 64, ([96, 160], [200, 56])), (8, 2, 128, ([300, 128, 1000], [1000, 420, 8]))])
def test_queued_training_steps_with_reused_buffers(tik, Hq, Hkv, d, lens):
    """Forward and backward of two batches in turn through the same lse, cu_seqlens and scratch: the dQ grid starts
    under the dK/dV grid without a wait of its own, and what it reads has to be this step's."""
    g = torch.Generator(device="cuda").manual_seed(11)
    tot, longest = sum(lens[0]), max(map(max, lens))
    assert sum(lens[1]) == tot
    data = [[torch.randn(tot, n, d, generator=g, device="cuda").to(torch.bfloat16) for n in (Hq, Hkv, Hkv, Hq)] for _ in lens]
    cus = [torch.tensor([0] + torch.tensor(x).cumsum(0).tolist(), dtype=torch.int32, device="cuda") for x in lens]
    bwd_ws = torch.empty(tik.workspace_bytes(tik.OP_ATTN_TRAIN_BWD, tot, Hq, Hkv, d), dtype=torch.uint8, device="cuda")
    lse, cu = torch.empty(tot, Hq, device="cuda"), cus[0].clone()

    def steps(sync):
        step = torch.cuda.synchronize if sync else (lambda: None)
        out = []
        for i in range(8):
            q, k, v, d_o = data[i % 2]
            cu.copy_(cus[i % 2]); step()
            o = tik.tik_attn_train_fwd(q, k, v, cu, longest, 0.1, lse=lse); step()
            out += [o, *tik.tik_attn_train_bwd(q, k, v, o, d_o, lse, cu, longest, 0.1, ws=bwd_ws)]; step()
        return out

    a, b = steps(True), steps(False)
    assert all(torch.equal(s, t) for s, t in zip(a, b))


def test_queued_long_prefills_with_a_reused_block_table(tik):
    """Contexts beyond 96 query tiles: the persistent grid fills the tail of the single-tile grid without a wait at
    its start, and reads the table of this call, written in place of the last one's."""
    Hq, Hkv, d, page, lens = 4, 1, 64, 64, [12500, 700]
    g = torch.Generator(device="cuda").manual_seed(12)
    blocks = -(-max(lens) // page)
    kc, vc = (torch.randn(2 * blocks, Hkv, page, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    tables = [torch.randperm(2 * blocks, generator=g, device="cuda").view(2, blocks).to(torch.int32) for _ in range(2)]
    q = torch.randn(sum(lens), Hq, d, generator=g, device="cuda").to(torch.bfloat16)
    ctx, cu = torch.tensor(lens, dtype=torch.int32, device="cuda"), torch.tensor([0, lens[0], sum(lens)], dtype=torch.int32, device="cuda")
    table = tables[0].clone()

    def calls(sync):
        step = torch.cuda.synchronize if sync else (lambda: None)
        out = []
        for i in range(6):
            table.copy_(tables[i % 2]); step()
            out.append(tik.tik_attn_prefill(q, cu, ctx, kc, vc, table, max(lens), max(lens), 0.1)); step()
        return out

    a, b = calls(True), calls(False)
    assert all(torch.equal(s, t) for s, t in zip(a, b)) and not torch.equal(a[0], a[1])
