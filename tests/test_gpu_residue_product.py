"""The product through residues (large layers) at the edges of its tiles: 256 rows on one side, a multiple of 32 on the other,
stages of 128 contraction indices in instructions of 32; and at the largest sums it may have to tell apart."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2505_07239_b200 import workloads as wl  # noqa: E402

U64 = np.uint64


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding

    return binding


R, L = "residue", "limb"


@pytest.fixture
def kernels(cb, monkeypatch):
    """The kernels of the products from here on, up and down in turn."""
    seen = []
    names = {cb.KERNEL_RESIDUE: R, cb.KERNEL_LIMB: L}
    for name in ("ffn_up", "ffn_down"):
        def call(ctx, tokens, original=getattr(cb.Comet, name)):
            original(ctx, tokens)
            seen.append(names.get(ctx.stats().product_kernel))

        monkeypatch.setattr(cb.Comet, name, call)
    return seen


@pytest.mark.parametrize("tokens,d_model,blocks,block,active,stacked,up,down", [
    (385, 1040, 80, 16, 63, 1, R, R),        # a row in the second token tile; depth 1040 = 8 stages and half an instruction;
                                             # columns of the weights' product on the 256-row side
    (257, 3088, 20, 48, 17, 1, R, R),        # strips of 48 columns; 816 of 1024 rows of the weights' tiles
    (400, 1552, 60, 16, 51, 1, R, R),        # 816 = 3 column tiles of 224 and a ragged one
    (449, 1040, 40, 32, 33, 2, R, L),        # two stacked matrices; the group boundary lies inside a tile; a weight side of
                                             # limbs opened beside a product through residues
    (417, 512, 60, 48, 56, 1, L, R),         # and the other way round
    (512, 1024, 40, 16, 32, 1, L, L),        # a layer just too small for it
])
def test_layer_at_tile_edges(cb, kernels, tokens, d_model, blocks, block, active, stacked, up, down):
    from tests import harness as hz

    cfg = wl.FFNConfig("residue-edges", tokens, d_model, blocks * block, block, 16, stacked == 2, active / blocks, "uniform",
                       "normal", "normal0.02", stacked=stacked)
    r = hz.run_and_compare_products(cfg, seed=800 + tokens, early_down=tokens != 400)
    assert r["mismatches"] == 0 and r["n_active"] == active * block, r
    assert kernels == [up, down]


@pytest.mark.parametrize("c_early", [False, True])
@pytest.mark.parametrize("T_up,T_down,up,down", [(300, 128, R, L), (128, 300, L, R)])
def test_weight_side_opened_for_another_number_of_tokens(cb, kernels, T_up, T_down, up, down, c_early):
    """comet_ffn_up opens the down-projection's weight side for the kernel that its own number of tokens asks for; comet_ffn_down
    with another number takes the other kernel and opens it again, whether C' was copied early or not."""
    import oracle

    d = n = 1536
    T = max(T_up, T_down)
    draw = lambda name, rows, cols: [wl.random_u64(31, f"other/{name}/{p}", rows * cols).reshape(rows, cols) for p in (0, 1)]  # noqa: E731
    W1, W2, B_up, B_dn = (draw(k, n, d) for k in ("W1", "W2", "B_up", "B_dn"))
    X, A_up, C_up = (draw(k, T_up, d) for k in ("X", "A_up", "C_up"))
    H, A_dn, C_dn = (draw(k, T_down, d) for k in ("H", "A_dn", "C_dn"))
    ctx = cb.Comet(T, d, n, 16, 16, 0, 0, n)
    keep = []

    def bind(tid, shares):
        for p in (0, 1):
            keep.append(cb.to_device(shares[p]))
            ctx.bind_shares(p, tid, keep[-1])

    bind(cb.W1, W1)
    bind(cb.W2, W2)
    assert ctx.set_mask(np.ones(n // 16, np.uint8)) == n
    if c_early:                                  # some C' of the up-projection's number of tokens, replaced below
        bind(cb.C_DN, draw("C_other", T_up, d))
    for tid, shares in ((cb.X, X), (cb.A_UP, A_up), (cb.B_UP, B_up), (cb.C_UP, C_up), (cb.B_DN, B_dn)):
        bind(tid, shares)
    ctx.ffn_up(T_up)
    t = lambda pair: [np.ascontiguousarray(m.T) for m in pair]  # noqa: E731  (stored output-feature-major)
    index = np.arange(n, dtype=np.int32)
    ref = oracle.somm(X, t(W1), index, A_up, t(B_up), C_up)
    for p in (0, 1):
        assert np.array_equal(ctx.get(p, cb.Z_UP, (T_up, n)), ref["Z"][p])
    for tid, shares in ((cb.H, H), (cb.A_DN, A_dn), (cb.C_DN, C_dn)):
        bind(tid, shares)
    ctx.ffn_down(T_down)
    ref = oracle.simm(H, t(W2), index, A_dn, t(B_dn), C_dn)
    for p in (0, 1):
        assert np.array_equal(ctx.get(p, cb.F_DN, (d, n)).T, ref["F"][p])
        assert np.array_equal(ctx.get(p, cb.Y, (T_down, d)), ref["Z"][p])
    assert kernels == [up, down]
    ctx.close()


def test_token_mask_of_one_component(cb):
    """Entries off the support under a token mask, against the CUDA-core path."""
    T, d, block, nab = 400, 1552, 16, 51
    n = block * nab
    mask = np.ones(nab, np.uint8)
    rng = np.random.default_rng(5)
    tmask = (rng.random((T, nab)) < 0.5).astype(np.uint8)
    tmask[:, 7] = 1                          # one block that every token uses: one component
    gen = torch.Generator(device="cuda").manual_seed(6)

    def pair(*shape):
        return [torch.randint(-(1 << 63), (1 << 63) - 1, shape, dtype=torch.int64, device="cuda", generator=gen) for _ in (0, 1)]

    shares = {cb.X: pair(T, d), cb.W1: pair(n, d), cb.W2: pair(d, n), cb.A_UP: pair(T, d), cb.B_UP: pair(n, d), cb.C_UP: pair(T, n),
              cb.H: pair(T, n), cb.A_DN: pair(T, n), cb.B_DN: pair(d, n), cb.C_DN: pair(T, d)}
    got = {}
    for path in (cb.PATH_LIMB, cb.PATH_SIMT):
        ctx = cb.Comet(T, d, n, block, 16, 0, 0, n, path)
        ctx.set_mask(mask)
        ctx.set_token_mask(tmask)
        for tid, s in shares.items():
            for p in (0, 1):
                ctx.load_shares(p, tid, s[p])
        ctx.ffn_up(T)
        kernels = [ctx.stats().product_kernel]
        ctx.ffn_down(T)
        kernels.append(ctx.stats().product_kernel)
        assert kernels == [cb.KERNEL_RESIDUE if path == cb.PATH_LIMB else cb.KERNEL_SIMT] * 2
        got[path] = [ctx.get(p, tid, s) for tid, s in ((cb.E_UP, (T, d)), (cb.Z_UP, (T, n)), (cb.E_DN, (T, n)), (cb.Y, (T, d)))
                     for p in (0, 1)]
        ctx.close()
    for a, b in zip(got[cb.PATH_LIMB], got[cb.PATH_SIMT]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("depth,residues", [(11424, True), (11440, False)])
def test_largest_sums(cb, depth, residues):
    """Every operand word of a row / column the same, so that Z_i = C_i + 2 * depth * e * f: words whose signed low 56 bits are
    the smallest and the largest there are put the sum at the bounds that the residues have to tell apart, up to the largest
    depth that goes through them."""
    words = np.array([0x0080000000000000, 0x007FFFFFFFFFFFFF, 0xFF80000000000000, 0x7F7FFFFFFFFFFFFF, 0xFFFFFFFFFFFFFFFF,
                      0x8000000000000000, 1, 0x8080808080808080, 0x00FF00FF00FF00FF, 0], dtype=U64)
    T, d = 512, 1024
    e, f = words[np.arange(T) * len(words) // T], words[np.arange(d) % len(words)]
    E, F = np.repeat(e[:, None], depth, 1), np.repeat(f[:, None], depth, 1)
    C = [wl.random_u64(9, f"largest/C{p}", T * d).reshape(T, d) for p in (0, 1)]
    ctx = cb.Comet(T, d, depth, 16, 16, 0, 0, depth)
    for p, (h, a, w, b) in enumerate(((E + E, E, F + F, F), (E * U64(0), E * U64(0), F, F))):
        ctx.load_shares(p, cb.W2, cb.to_device(w))
        if p == 0:
            assert ctx.set_mask(np.ones(depth // 16, np.uint8)) == depth
        for tid, s in ((cb.H, h), (cb.A_DN, a), (cb.B_DN, b), (cb.C_DN, C[p])):
            ctx.load_shares(p, tid, cb.to_device(s))
    ctx.ffn_down(T)
    assert (ctx.stats().product_kernel == cb.KERNEL_RESIDUE) == residues
    want = U64(2 * depth) * (e[:, None] * f[None, :])
    for p in (0, 1):
        assert np.array_equal(ctx.get(p, cb.Y, (T, d)), C[p] + want), p
    ctx.close()


@pytest.mark.parametrize("T,n", [(2550, 12304), (2100, 14864)])       # rows of Z on the 256-row side, columns of Z on it
def test_more_residues_than_the_scratch_holds(cb, T, n):
    """Two bands, the second one ragged, against the CUDA-core path."""
    d, block = 528, 16
    gen = torch.Generator(device="cuda").manual_seed(T)

    def pair(*shape):
        return [torch.randint(-(1 << 63), (1 << 63) - 1, shape, dtype=torch.int64, device="cuda", generator=gen) for _ in (0, 1)]

    shares = {cb.X: pair(T, d), cb.W1: pair(n, d), cb.A_UP: pair(T, d), cb.B_UP: pair(n, d), cb.C_UP: pair(T, n)}
    got = []
    for path in (cb.PATH_AUTO, cb.PATH_SIMT):
        ctx = cb.Comet(T, d, n, block, 16, 0, 0, n, path)
        ctx.set_mask(np.ones(n // block, np.uint8))
        for tid, s in shares.items():
            for p in (0, 1):
                ctx.bind_shares(p, tid, s[p])
        before = ctx.stats().kernel_launches
        ctx.ffn_up(T)
        if path == cb.PATH_AUTO:                 # the exchange, then product and recombination of either band
            assert ctx.stats().product_kernel == cb.KERNEL_RESIDUE and ctx.stats().kernel_launches == before + 5
        ctx.synchronize()
        got.append([ctx.result_view(p, cb.Z_UP, (T, n)).clone() for p in (0, 1)])
        torch.cuda.synchronize()
        ctx.close()
    for p in (0, 1):
        assert torch.equal(got[0][p], got[1][p]), p


@pytest.mark.parametrize("stays_free,residues", [(0.30, True), (0.20, False)])
def test_room_for_residues_leaves_memory_free(cb, stays_free, residues):
    """A quarter of the device's memory has to stay free for a context to take room for residues; the others multiply through
    limbs, in less memory, and leave the same bits."""
    T, d, n, block = 512, 1536, 1536, 16
    gen = torch.Generator(device="cuda").manual_seed(8)
    shares = {t: [torch.randint(-(1 << 63), (1 << 63) - 1, s, dtype=torch.int64, device="cuda", generator=gen) for _ in (0, 1)]
              for t, s in ((cb.X, (T, d)), (cb.W1, (n, d)), (cb.A_UP, (T, d)), (cb.B_UP, (n, d)), (cb.C_UP, (T, n)))}

    def product():
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = cb.Comet(T, d, n, block, 16, 0, 0, n)
        taken = before - torch.cuda.mem_get_info()[0]
        ctx.set_mask(np.ones(n // block, np.uint8))
        for tid, s in shares.items():
            for p in (0, 1):
                ctx.bind_shares(p, tid, s[p])
        ctx.ffn_up(T)
        ctx.synchronize()
        out = [ctx.result_view(p, cb.Z_UP, (T, n)).clone() for p in (0, 1)]
        kernel = ctx.stats().product_kernel
        torch.cuda.synchronize()
        ctx.close()
        return out, kernel, taken

    torch.cuda.empty_cache()
    product()                                    # loads what there is to load
    want, kernel, most = product()
    assert kernel == cb.KERNEL_RESIDUE
    free, everything = torch.cuda.mem_get_info()
    held = torch.empty(free - int(stays_free * everything), dtype=torch.uint8, device="cuda")     # never written
    got, kernel, taken = product()
    del held
    torch.cuda.empty_cache()
    assert kernel == (cb.KERNEL_RESIDUE if residues else cb.KERNEL_LIMB)
    assert (taken < 0.8 * most) == (not residues), (taken, most)
    assert all(torch.equal(a, b) for a, b in zip(want, got))


def test_captured_and_replayed(cb, kernels):
    from tests.test_gpu_capture import test_layer_captured_and_replayed as replayed

    replayed(cb, 385, 1040, 80, 16, 63)
    assert set(kernels) == {R}


@pytest.mark.parametrize("x_on", ["Y", "Z_UP"])
def test_operands_on_result_buffers(cb, kernels, x_on):
    from tests.test_gpu_bound_results import test_operands_on_result_buffers as bound

    bound(385, 1040, x_on)
    assert set(kernels) == {R}
