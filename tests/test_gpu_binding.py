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
