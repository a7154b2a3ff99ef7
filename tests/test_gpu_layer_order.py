"""The order of a context's work on its stream, the projections of a layer apart from each other: graphs of either alone, and layers back
to back with nothing read in between.  Bit for bit against the CPU oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from tests.test_gpu_capture import _Layer  # noqa: E402


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding

    return binding


class _Parts(_Layer):
    def enqueue_up(self):
        cb, ctx = self.cb, self.ctx
        assert ctx.set_mask(self.mask) == self.n
        for t, pair in self.buffers.items():
            for p in (0, 1):
                ctx.bind_shares(p, t, pair[p])
        ctx.ffn_up(self.T)

    def products(self, v):
        cb, t = self.cb, lambda pair: [np.ascontiguousarray(m.T) for m in pair]  # noqa: E731  (stored output-feature-major)
        return (oracle.somm(v[cb.X], t(self.W[cb.W1]), self.I, v[cb.A_UP], t(v[cb.B_UP]), v[cb.C_UP])["Z"],
                oracle.simm(v[cb.H], t(self.W[cb.W2]), self.I, v[cb.A_DN], t(v[cb.B_DN]), v[cb.C_DN])["Z"])

    def results(self):
        return [self.ctx.result_view(p, t, (self.T, cols)) for t, cols in ((self.cb.Z_UP, self.n), (self.cb.Y, self.d)) for p in (0, 1)]

    def check_results(self, v):
        """The results alone: they can be read where a replay has written them."""
        self.ctx.synchronize()
        for got, want in zip(self.results(), (z for pair in self.products(v) for z in pair)):
            assert np.array_equal(got.cpu().numpy().view(np.uint64), want)


@pytest.mark.parametrize("tokens,d,blocks,block,active", [
    (128, 304, 32, 16, 28),                                # the down-projection's weight side in the launch before the product
    (200, 960, 24, 16, 16), (512, 1024, 24, 16, 14),       # beside it: few words, and a long product
])
@pytest.mark.parametrize("up_captured", [True, False])
def test_projections_captured_apart(cb, tokens, d, blocks, block, active, up_captured):
    """A graph of the down-projection alone, behind a graph of the up-projection or an ordinary call of it: the functionality
    between the two is the caller's."""
    layer = _Parts(cb, tokens, d, blocks, block, active)
    layer.fill(1)
    layer.enqueue()
    layer.stream.synchronize()
    graphs = [torch.cuda.CUDAGraph() for _ in (0, 1)]
    if up_captured:
        with torch.cuda.graph(graphs[0], stream=layer.stream):
            layer.enqueue_up()
    else:
        layer.enqueue_up()
        layer.stream.synchronize()
    with torch.cuda.graph(graphs[1], stream=layer.stream):
        layer.ctx.ffn_down(tokens)
    for step in (2, 3):
        v = layer.fill(step)
        with torch.cuda.stream(layer.stream):
            if up_captured:
                graphs[0].replay()
            else:
                layer.enqueue_up()
            graphs[1].replay()
        (layer.check if up_captured else layer.check_results)(v)
    del graphs
    layer.ctx.close()


@pytest.mark.parametrize("tokens,d,blocks,block,active,kernel", [
    (16, 256, 32, 32, 3, "KERNEL_STREAM"), (32, 256, 32, 32, 3, "KERNEL_STREAM"),        # tiles of 32 features
    (32, 1008, 64, 16, 49, "KERNEL_STREAM"),                                             # of 128
    (128, 304, 32, 16, 28, "KERNEL_LIMB"), (512, 1024, 24, 16, 14, "KERNEL_LIMB"),       # tiles in parts; a launch beside the product
])
def test_layers_back_to_back(cb, tokens, d, blocks, block, active, kernel):
    """Product, truncation, product, truncation, pass after pass and nothing in between: a kernel's CTAs are set up while the kernels
    before it are still at work.  The inputs of each pass are bound where they lie."""
    layer = _Parts(cb, tokens, d, blocks, block, active)
    ctx = layer.ctx
    inputs = [{t: layer._draw(step, f"in{t}", s) for t, s in layer.shapes.items()} for step in range(4)]
    resident = [{t: [cb.to_device(x) for x in pair] for t, pair in v.items()} for v in inputs]
    views = layer.results()
    torch.cuda.synchronize()
    kept = []
    with torch.cuda.stream(layer.stream):
        for step in range(24):
            ctx.set_mask(layer.mask)
            for t, pair in resident[step % 4].items():
                for p in (0, 1):
                    ctx.bind_shares(p, t, pair[p])
            ctx.ffn_up(tokens)
            ctx.truncate(cb.Z_UP)
            ctx.ffn_down(tokens)
            ctx.truncate(cb.Y)
            if step >= 20:                             # the first of them after 21 passes without anything else
                kept.append([v.clone() for v in views])
    assert ctx.stats().product_kernel == getattr(cb, kernel)
    ctx.synchronize()
    for v, got in zip(inputs, kept):
        want = [oracle.truncate(p, pair[p], 16) for pair in layer.products(v) for p in (0, 1)]
        for g, w in zip(got, want):
            assert np.array_equal(g.cpu().numpy().view(np.uint64), w)
    ctx.close()
