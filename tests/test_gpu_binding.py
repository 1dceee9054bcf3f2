"""The extension module behind binding.py: outputs made or given, refused arguments, threads on streams of their own."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tik():
    from paper_2609_35140_b200 import binding
    binding.load()
    yield binding
    assert binding.device_status() == 0


def _x(rows, cols, seed, std=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(rows, cols, generator=g, device="cuda") * std).to(torch.bfloat16)


def test_given_output_is_returned_and_equals_a_made_one(tik):
    x, w = _x(33, 256, 1), _x(72, 256, 2, 0.05)
    y = torch.full((33, 72), 7.0, dtype=torch.bfloat16, device="cuda")
    assert tik.tik_linear(x, w, y=y) is y
    assert torch.equal(y, tik.tik_linear(x, w))
    out = torch.empty(33, 128, dtype=torch.bfloat16, device="cuda")
    assert tik.tik_swiglu(x, out) is out
    ws = torch.empty(tik.workspace_bytes(tik.OP_TOKEN_LOGPROB, 33, H=256, V=72), dtype=torch.uint8, device="cuda")
    ids, lse = torch.arange(33, dtype=torch.int32, device="cuda"), torch.empty(33, device="cuda")
    a = tik.tik_token_logprob(x, w, ids, 1, ws=ws, lse=lse)
    assert torch.equal(a, tik.tik_token_logprob(x, w, ids)) and bool((lse > a).all())


def test_refused_arguments(tik):
    x, w = _x(8, 128, 3), _x(16, 128, 4)
    for bad in (lambda: tik.tik_linear(x.float(), w), lambda: tik.tik_linear(x.t(), w), lambda: tik.tik_linear(x.cpu(), w),
                lambda: tik.tik_linear(x[:, :100].contiguous(), w),
                lambda: tik.tik_token_logprob(x, w, torch.zeros(8, dtype=torch.int64, device="cuda")),
                lambda: tik.tik_token_logprob(x, w, torch.zeros(8, dtype=torch.int32, device="cuda"),
                                              ws=torch.empty(16, dtype=torch.uint8, device="cuda"))):
        with pytest.raises(tik.TikError):
            bad()
    with pytest.raises(ValueError):
        tik.tik_attn_train_fwd(x, w, w, torch.zeros(2, dtype=torch.int32, device="cuda"), 8, 0.1)
    with pytest.raises(TypeError):
        tik.tik_linear(3, w)


def test_tensors_without_the_axis_that_is_read_are_refused(tik):
    """A size is read, and refused, before the interpreter lock is dropped for the call: an exception behind that
    point would end the process instead of raising."""
    i32 = lambda *v: torch.tensor(v, dtype=torch.int32, device="cuda")
    q, k, scalar = (torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in ((2, 4, 64), (2, 1, 64), ()))
    cache, table = torch.zeros(2, 1, 16, 64, dtype=torch.bfloat16, device="cuda"), i32(0, 1).view(2, 1)
    rope, weight = torch.zeros(8, 64, device="cuda"), torch.ones(64, dtype=torch.bfloat16, device="cuda")
    for bad in (lambda: tik.tik_kv_cache_write(scalar, scalar, i32(0, 1), i32(1), cache, cache, table),
                lambda: tik.tik_kv_cache_write(k, k, i32(0, 1, 2), i32(1, 1), cache, cache, i32(0, 1)),
                lambda: tik.tik_qk_norm_rope_kv_write(q, k, k, weight, weight, 1e-6, rope[0, 0].clone(), i32(0, 1, 2)),
                lambda: tik.tik_qk_norm_rope_kv_write(q, scalar, k, weight, weight, 1e-6, rope, i32(0, 1, 2)),
                lambda: tik.tik_qk_norm_rope_kv_write(q, k, k, weight, weight, 1e-6, rope, i32(0, 1, 2), i32(1, 1), scalar,
                                                      cache, table),
                lambda: tik.tik_linear(q[0], scalar), lambda: tik.tik_attn_train_fwd(q, scalar, scalar, i32(0, 2), 2, 0.1)):
        with pytest.raises(IndexError):
            bad()
    assert bool((cache == 0).all())


def test_threads_with_streams_of_their_own(tik):
    w = _x(640, 512, 5, 0.05)
    xs = [_x(40 + i, 512, 6 + i) for i in range(4)]
    want = [tik.tik_linear(x, w) for x in xs]
    torch.cuda.synchronize()
    got = [None] * len(xs)

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(50):
                got[i] = tik.tik_linear(xs[i], w)
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(xs))]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert all(torch.equal(a, b) for a, b in zip(got, want))
