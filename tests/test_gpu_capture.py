"""The order of a context's work on its stream.  Calls captured in a CUDA graph: a layer captured once, an ordinary step before
the first replay, replays with new inputs in the bound buffers, and an ordinary step after them; an index list.  A context
made while the default stream is busy.  Bit for bit against the CPU oracle."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2505_07239_b200 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding

    return binding


class _Layer:
    """One layer of one weight matrix on a stream of its own, every input bound to a buffer that is refilled per step."""

    def __init__(self, cb, tokens, d, blocks, block, active):
        self.cb, self.T, self.d, self.n, D = cb, tokens, d, active * block, blocks * block
        self.stream = torch.cuda.Stream()
        self.ctx = cb.Comet(tokens, d, D, block, 16, max_active=self.n, stream=self.stream)
        self.mask = np.zeros(blocks, np.uint8)
        self.mask[np.random.default_rng(tokens).permutation(blocks)[:active]] = 1
        self.I = oracle.index_set(self.mask, block, 1)
        self.W = {t: self._draw(0, f"W{t}", s) for t, s in ((cb.W1, (D, d)), (cb.W2, (d, D)))}
        self.weights = {t: [cb.to_device(w) for w in pair] for t, pair in self.W.items()}
        n = self.n
        self.shapes = {cb.X: (tokens, d), cb.A_UP: (tokens, d), cb.B_UP: (n, d), cb.C_UP: (tokens, n), cb.H: (tokens, n),
                       cb.A_DN: (tokens, n), cb.B_DN: (d, n), cb.C_DN: (tokens, d)}
        self.buffers = {t: [torch.zeros(s, dtype=torch.int64, device="cuda") for _ in (0, 1)] for t, s in self.shapes.items()}
        torch.cuda.synchronize()
        for t, pair in self.weights.items():
            for p in (0, 1):
                self.ctx.bind_shares(p, t, pair[p])

    def _draw(self, step, name, shape):
        return [wl.random_u64(50 + self.T + step, f"capture/{name}/{p}", shape[0] * shape[1]).reshape(shape) for p in (0, 1)]

    def fill(self, step):
        """New inputs into the buffers, on the stream; returns them."""
        v = {t: self._draw(step, f"in{t}", s) for t, s in self.shapes.items()}
        with torch.cuda.stream(self.stream):
            for t, pair in v.items():
                for p in (0, 1):
                    self.buffers[t][p].copy_(torch.from_numpy(pair[p].view(np.int64)))
        return v

    def enqueue(self):
        cb, ctx = self.cb, self.ctx
        assert ctx.set_mask(self.mask) == self.n
        for t, pair in self.buffers.items():
            for p in (0, 1):
                ctx.bind_shares(p, t, pair[p])
        ctx.ffn_up(self.T)
        ctx.ffn_down(self.T)

    def check(self, v):
        cb, (W1, W2) = self.cb, (self.W[self.cb.W1], self.W[self.cb.W2])
        t = lambda pair: [np.ascontiguousarray(m.T) for m in pair]  # noqa: E731  (stored output-feature-major)
        up = oracle.somm(v[cb.X], t(W1), self.I, v[cb.A_UP], t(v[cb.B_UP]), v[cb.C_UP])
        down = oracle.simm(v[cb.H], t(W2), self.I, v[cb.A_DN], t(v[cb.B_DN]), v[cb.C_DN])
        self.ctx.synchronize()
        for p in (0, 1):
            for ref, ids, rows, cols in ((up, (cb.E_UP, cb.F_UP, cb.Z_UP), self.n, self.d),
                                         (down, (cb.E_DN, cb.F_DN, cb.Y), self.d, self.n)):
                assert np.array_equal(self.ctx.get(p, ids[0], (self.T, cols)), ref["E"][p])
                assert np.array_equal(self.ctx.get(p, ids[1], (rows, cols)).T, ref["F"][p])
                assert np.array_equal(self.ctx.get(p, ids[2], (self.T, rows)), ref["Z"][p])


@pytest.mark.parametrize("tokens,d,blocks,block,active", [
    (16, 144, 24, 16, 9), (32, 144, 24, 16, 9),        # the streaming kernel: one token tile
    (48, 1024, 64, 16, 48),                            # two token tiles
    (48, 272, 24, 16, 9), (70, 1024, 24, 16, 17),      # exchange and tensor-core kernel: one stream, and with the side stream
])
def test_layer_captured_and_replayed(cb, tokens, d, blocks, block, active):
    layer = _Layer(cb, tokens, d, blocks, block, active)
    layer.fill(1)
    layer.enqueue()                                    # first use outside the capture
    layer.stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=layer.stream):
        layer.enqueue()
    v = layer.fill(2)
    layer.enqueue()                                    # captured but not yet run, an ordinary step in between
    layer.check(v)
    for step in (3, 4, 5):
        v = layer.fill(step)
        with torch.cuda.stream(layer.stream):
            graph.replay()
        layer.check(v)
    v = layer.fill(6)
    layer.enqueue()
    layer.check(v)
    del graph
    layer.ctx.close()


@pytest.mark.parametrize("blocks", [1, 1024, 1040])    # lists that travel with the launches, and one that a kernel compacts
def test_index_list_captured_and_replayed(cb, blocks):
    stream = torch.cuda.Stream()
    ctx = cb.Comet(4, 16, blocks * 16, 16, 12, stream=stream)
    rng = np.random.default_rng(blocks)
    masks = [(rng.random(blocks) < 0.5).astype(np.uint8) for _ in range(3)]
    masks[1][-1] = 1
    out = torch.full((blocks,), -1, dtype=torch.int32, device="cuda")
    count = ctypes.c_int32()
    ctx.set_mask(masks[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.set_mask(masks[1])
        assert cb.library().comet_get_index(ctx._h, out.data_ptr(), cb.DEVICE, blocks, ctypes.byref(count)) == cb.OK
    ctx.set_mask(masks[2])                             # what the list was taken from is gone
    for _ in range(2):
        out.fill_(-1)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        assert out[:count.value].tolist() == np.flatnonzero(masks[1]).tolist()
        assert (out[count.value:] == -1).all()
    host = np.full(blocks, -1, np.int32)
    ctx.set_mask(masks[2])
    assert cb.library().comet_get_index(ctx._h, host.ctypes.data, cb.HOST, blocks, ctypes.byref(count)) == cb.OK
    ctx.synchronize()
    assert host[:count.value].tolist() == np.flatnonzero(masks[2]).tolist()
    del graph
    ctx.close()


def test_context_made_while_the_default_stream_is_busy(cb):
    """The words that the kernels count in are cleared in the order of the context's own stream."""
    mask = np.zeros(24, np.uint8)
    mask[3:12] = 1
    stream = torch.cuda.Stream()
    for cycles in (0, 200_000_000):                    # a first pass that loads what there is to load, then a tenth of a second
        torch.cuda.synchronize()
        if cycles:
            torch.cuda._sleep(cycles)                  # on the default stream
        with torch.cuda.stream(stream):
            ctx = cb.Comet(16, 144, 384, 16, 16, max_active=144, stream=stream)
            X, A, B, C = (torch.zeros(s, dtype=torch.int64, device="cuda") for s in ((16, 144), (16, 144), (144, 144), (16, 144)))
            W = torch.zeros((384, 144), dtype=torch.int64, device="cuda")
            C.fill_(5)
            assert ctx.set_mask(mask) == 144
            for p in (0, 1):
                for t, v in ((cb.W1, W), (cb.X, X), (cb.A_UP, A), (cb.B_UP, B), (cb.C_UP, C)):
                    ctx.bind_shares(p, t, v)
            ctx.ffn_up(16)
            out = [ctx.result_view(p, cb.Z_UP, (16, 144)).clone() for p in (0, 1)]
            stream.synchronize()
            # the product ran while the default stream was still at work: the case that is meant
            assert not cycles or not torch.cuda.default_stream().query()
        ctx.synchronize()
        assert all(bool((z == 5).all()) for z in out)
        torch.cuda.synchronize()
        ctx.close()
