"""Inputs bound to the library's own result buffers: X to the result of the layer before, X and H to the buffer that the same call
writes.  Bit for bit against the CPU oracle, through the streaming kernel and through the exchange."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2505_07239_b200 import workloads as wl  # noqa: E402


@pytest.mark.parametrize("x_on", ["Y", "Z_UP"])
@pytest.mark.parametrize("tokens,d", [(16, 144), (48, 144), (130, 496), (70, 528)])   # the last: weight side on its own stream
def test_operands_on_result_buffers(tokens, d, x_on):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding as cb

    block, D = 16, 2 * d
    mask = np.zeros(D // block, np.uint8)
    mask[1::2] = 1                                     # n = d, so that every result has X's and H's shape
    index = oracle.index_set(mask, block, 1)
    n, T = index.size, tokens
    assert n == d
    draw = lambda k, *s: [wl.random_u64(60 + T, f"bound/{k}/{p}", s[0] * s[1]).reshape(s) for p in (0, 1)]  # noqa: E731
    shapes = {cb.W1: (D, d), cb.W2: (d, D), cb.A_UP: (T, d), cb.B_UP: (n, d), cb.C_UP: (T, n), cb.A_DN: (T, n),
              cb.B_DN: (d, n), cb.C_DN: (T, d)}
    v = {k: draw(k, *s) for k, s in shapes.items()}
    stream = torch.cuda.Stream()
    ctx = cb.Comet(T, d, D, block, 16, max_active=n, stream=stream)
    assert ctx.set_mask(mask) == n
    dev = {k: [cb.to_device(w) for w in pair] for k, pair in v.items()}
    torch.cuda.synchronize()
    place = {"Y": cb.Y, "Z_UP": cb.Z_UP}[x_on]
    x_view = [ctx.result_view(p, place, (T, d)) for p in (0, 1)]
    h_view = [ctx.result_view(p, cb.Y, (T, n)) for p in (0, 1)]
    t = lambda pair: [np.ascontiguousarray(m.T) for m in pair]  # noqa: E731  (stored output-feature-major)
    for k, pair in dev.items():
        for p in (0, 1):
            if k != cb.C_DN:
                ctx.bind_shares(p, k, pair[p])

    def into(views, name):
        w = draw(name, T, d)
        with torch.cuda.stream(stream):
            for p in (0, 1):
                views[p].copy_(torch.from_numpy(w[p].view(np.int64)))
        return w

    for step in range(3):
        X = into(x_view, f"X{step}")
        for p in (0, 1):
            if step == 0:
                ctx.bind_shares(p, cb.X, x_view[p])    # later steps: still bound, new contents
            ctx.load_shares(p, cb.C_DN, dev[cb.C_DN][p])
        ctx.ffn_up(T)
        up = oracle.somm(X, t(v[cb.W1]), index, v[cb.A_UP], t(v[cb.B_UP]), v[cb.C_UP])
        for p in (0, 1):
            assert np.array_equal(ctx.get(p, cb.E_UP, (T, d)), up["E"][p])
            assert np.array_equal(ctx.get(p, cb.Z_UP, (T, n)), up["Z"][p])
        H = into(h_view, f"H{step}")
        for p in (0, 1):
            ctx.bind_shares(p, cb.H, h_view[p])
            ctx.load_shares(p, cb.C_DN, dev[cb.C_DN][p])   # Y holds H now, not what was copied there early
        ctx.ffn_down(T)
        down = oracle.simm(H, t(v[cb.W2]), index, v[cb.A_DN], t(v[cb.B_DN]), v[cb.C_DN])
        for p in (0, 1):
            assert np.array_equal(ctx.get(p, cb.E_DN, (T, n)), down["E"][p])
            assert np.array_equal(ctx.get(p, cb.Y, (T, d)), down["Z"][p])
    ctx.close()


@pytest.mark.parametrize("on_y", ["C_UP", "X"])
def test_operand_on_y_while_c_may_be_copied_there(on_y):
    """The up-projection through residues, which reads its C share after the product, and the down-projection through limbs,
    whose C' is copied into Y beside the up-projection when it is loaded by then."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding as cb

    T, d, block, blocks, g = 385, 2064, 16, 36, 2
    D, n = blocks * block, 30 * block
    mask = np.ones(blocks, np.uint8)
    mask[3::6] = 0
    index, index_up = oracle.index_set(mask, block, 1), oracle.index_set(mask, block, g)
    shapes = {cb.X: (T, d), cb.W1: (D, d), cb.WG: (D, d), cb.W2: (d, D), cb.A_UP: (T, d), cb.B_UP: (g * n, d), cb.C_UP: (T, g * n),
              cb.H: (T, n), cb.A_DN: (T, n), cb.B_DN: (d, n), cb.C_DN: (T, d)}
    v = {k: [wl.random_u64(71, f"on_y/{k}/{p}", s[0] * s[1]).reshape(s) for p in (0, 1)] for k, s in shapes.items()}
    dev = {k: [cb.to_device(w) for w in pair] for k, pair in v.items()}
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = cb.Comet(T, d, D, block, 16, g - 1, max_active=n, stream=stream)
    assert ctx.set_mask(mask) == n
    on = {"C_UP": cb.C_UP, "X": cb.X}[on_y]
    for k, pair in dev.items():
        for p in (0, 1):
            share = pair[p]
            if k == on:
                share = ctx.result_view(p, cb.Y, shapes[k])
                with torch.cuda.stream(stream):
                    share.copy_(pair[p])
            ctx.bind_shares(p, k, share)
    t = lambda pair: [np.ascontiguousarray(m.T) for m in pair]  # noqa: E731  (stored output-feature-major)
    ctx.ffn_up(T)
    assert ctx.stats().product_kernel == cb.KERNEL_RESIDUE
    W = [np.concatenate([v[cb.WG][p], v[cb.W1][p]]) for p in (0, 1)]
    up = oracle.somm(v[cb.X], t(W), index_up, v[cb.A_UP], t(v[cb.B_UP]), v[cb.C_UP])
    for p in (0, 1):
        assert np.array_equal(ctx.get(p, cb.E_UP, (T, d)), up["E"][p])
        assert np.array_equal(ctx.get(p, cb.Z_UP, (T, g * n)), up["Z"][p])
    ctx.ffn_down(T)
    assert ctx.stats().product_kernel == cb.KERNEL_LIMB
    down = oracle.simm(v[cb.H], t(v[cb.W2]), index, v[cb.A_DN], t(v[cb.B_DN]), v[cb.C_DN])
    for p in (0, 1):
        assert np.array_equal(ctx.get(p, cb.E_DN, (T, n)), down["E"][p])
        assert np.array_equal(ctx.get(p, cb.Y, (T, d)), down["Z"][p])
    ctx.close()
