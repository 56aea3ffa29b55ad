"""Calls on a stream other than the current one: their inputs are produced, and their outputs allocated, on the
current stream.  The delays make a missing wait show as wrong values."""
import numpy as np
import pytest

from paper_2410_05911_gb300 import aecct as A
from paper_2410_05911_gb300 import inputs as I

torch = pytest.importorskip("torch")

DELAY = 100_000_000  # cycles, about 50 ms


def same(got, want):
    return all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want))


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["contiguous", "transposed", "half"])
def test_ternarize_on_another_stream(form):
    rng = np.random.Generator(np.random.PCG64(7))
    host = [torch.from_numpy(rng.standard_normal((64, 128)).astype(np.float32)).cuda() for _ in range(5)]
    if form == "half":
        host = [t.half() for t in host]
    view = (lambda t: t.t()) if form == "transposed" else (lambda t: t)
    codes, scale, wq = A.aap_ternarize([view(t) for t in host], want_weights=True)
    want = [*codes, scale, *wq]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    # the weights are written on the current stream, late
    w = [torch.zeros_like(t) for t in host]
    torch.cuda._sleep(DELAY)
    for a, b in zip(w, host):
        a.copy_(b)
    codes, scale, wq = A.aap_ternarize([view(t) for t in w], want_weights=True, stream=side)
    side.synchronize()
    assert same([*codes, scale, *wq], want)
    # the weights and the outputs go back to the allocator while the other stream has not begun
    with torch.cuda.stream(side):
        torch.cuda._sleep(DELAY)
    codes, scale, wq = A.aap_ternarize([view(t) for t in w], want_weights=True, stream=side)
    shapes = [t.shape for t in w]
    del w
    other = [torch.full(s, 7.0, device="cuda") for s in shapes for _ in range(4)]
    torch.cuda.current_stream().synchronize()
    side.synchronize()
    assert same([*codes, scale, *wq], want)
    del codes, scale, wq
    assert all(bool((t == 7.0).all()) for t in other)


@pytest.mark.gpu
@pytest.mark.parametrize("strided", [False, True])
def test_decode_on_another_stream(strided):
    model = I.random_model(I.make_code("polar64_32"), 64, 2, seed=3, spe_noise=True)
    dec = A.Decoder(model)
    host = torch.from_numpy(np.random.Generator(np.random.PCG64(9)).standard_normal((300, 64)).astype(np.float32)).cuda()
    want = [t.clone() for t in dec.decode(host)]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()

    def late(value):
        y = torch.zeros((300, 128 if strided else 64), device="cuda")
        torch.cuda._sleep(DELAY)
        part = y[:, ::2] if strided else y
        part.copy_(value)
        return part

    got = dec.decode(late(host), stream=side)
    side.synchronize()
    assert same(got, want)
    # the words go back to the allocator while the other stream has not begun
    y = late(host)
    with torch.cuda.stream(side):
        torch.cuda._sleep(DELAY)
    got = dec.decode(y, stream=side)
    del y
    other = [torch.full((300, 128 if i else 64), 7.0, device="cuda") for i in range(4)]
    torch.cuda.current_stream().synchronize()
    side.synchronize()
    assert same(got, want)
    del got
    assert all(bool((t == 7.0).all()) for t in other)
    assert dec.synchronize() == A.AECCT_OK
    dec.close()


@pytest.mark.gpu
def test_decode_captured_on_a_stream_that_is_not_current():
    model = I.random_model(I.make_code("bch31_16"), 32, 2, seed=3, spe_noise=True)
    dec = A.Decoder(model)
    y = torch.from_numpy(np.random.Generator(np.random.PCG64(9)).standard_normal((40, 31)).astype(np.float32)).cuda()
    want = [t.clone() for t in dec.decode(y)]
    out = [torch.empty_like(t) for t in want]
    torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK  # no status query is left for the captured call
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        graph.capture_begin()
    dec.decode(y, out=out, stream=side)  # the current stream is not under capture
    with torch.cuda.stream(side):
        graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    assert same(out, want)
    dec.close()
