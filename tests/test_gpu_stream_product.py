"""The streaming product kernel (few token rows; the allocation-free entry point) at the edges of its tiles: 32 tokens,
128 output features in quarters of 32, steps of 32 contraction indices.  Bit for bit against the CPU oracle."""
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


@pytest.mark.parametrize("T,K,N", [
    (1, 8, 4),             # the smallest problem: one step, one quarter, a quarter of a step deep
    (3, 40, 28), (32, 32, 32), (33, 64, 36),      # one and two token tiles
    (16, 72, 160), (17, 72, 160),                 # accumulators of 16 and 32 columns
    (31, 104, 128), (65, 96, 132),                # a full feature tile, and four features into the next
    (7, 1032, 420),        # more steps than SMs in one tile's range, ragged in every direction
    (1, 16, 32752),        # 256 feature tiles of a single step: the scratch array's limit in N
    (2000, 32, 4),         # 63 token tiles against four features
    (14208, 8, 64), (14209, 8, 64), (14209, 8, 68), (14209, 16, 64), (65531, 8, 4),    # both sides of what the CUDA cores take
    (2, 65536, 4),         # a single tile 2048 steps deep: more than one segment's bound on the contraction depth
])
def test_static_product_at_tile_edges(cb, T, K, N):
    def draw(name, shape):
        return [wl.random_u64(900 + T, f"stream/{name}/{p}", shape[0] * shape[1]).reshape(shape) for p in (0, 1)]

    Xh, Ah, Yh, Bh, Ch = draw("X", (T, K)), draw("A", (T, K)), draw("Y", (N, K)), draw("B", (N, K)), draw("C", (T, N))
    X, A, Y, B, C = ([cb.to_device(v) for v in pair] for pair in (Xh, Ah, Yh, Bh, Ch))
    Z = [torch.full((T, N), -1, dtype=torch.int64, device="cuda") for _ in (0, 1)]
    assert cb.beaver_matmul_static(X, A, Y, B, C, Z) == cb.OK
    torch.cuda.synchronize()
    ref = oracle.pi_matmul(Xh, [np.ascontiguousarray(v.T) for v in Yh], Ah, [np.ascontiguousarray(v.T) for v in Bh], Ch)
    for p in (0, 1):
        assert np.array_equal(Z[p].cpu().numpy().view(np.uint64), ref["Z"][p]), p


@pytest.mark.parametrize("on", ["X", "Y", "C"])
@pytest.mark.parametrize("T,K,N", [(8, 8, 8), (64, 64, 64), (200, 200, 200)])
def test_static_product_in_place(cb, T, K, N, on):
    """The result on the memory of an operand of the same size."""
    v = {k: [wl.random_u64(950 + T, f"place/{k}/{p}", s[0] * s[1]).reshape(s) for p in (0, 1)]
         for k, s in {"X": (T, K), "A": (T, K), "Y": (N, K), "B": (N, K), "C": (T, N)}.items()}
    d = {k: [cb.to_device(w) for w in pair] for k, pair in v.items()}
    assert cb.beaver_matmul_static(d["X"], d["A"], d["Y"], d["B"], d["C"], d[on]) == cb.OK
    torch.cuda.synchronize()
    ref = oracle.pi_matmul(v["X"], [np.ascontiguousarray(w.T) for w in v["Y"]], v["A"],
                           [np.ascontiguousarray(w.T) for w in v["B"]], v["C"])
    for p in (0, 1):
        assert np.array_equal(d[on][p].cpu().numpy().view(np.uint64), ref["Z"][p]), p


@pytest.mark.parametrize("tokens,d_model,blocks,block,active,stacked,streamed", [
    (1, 16, 4, 16, 1, 1, True),          # 16 features, half a step
    (32, 144, 24, 16, 9, 1, True),       # 144 features both ways: 128 and a ragged tile of 16
    (31, 112, 12, 48, 5, 2, True),       # strips of 48 columns: a step takes its halves from two blocks
    (8, 272, 8, 80, 3, 3, True),         # three stacked matrices, group boundaries inside a feature tile
    (16, 1184, 16, 16, 8, 1, True), (17, 1184, 16, 16, 8, 1, True),        # 4 x 37 steps of tiles of 32 features, 37 x 4: all at once
    (17, 1200, 16, 16, 8, 1, True),      # .. and 4 x 38 of the one side, 38 x 4 of the other: tiles of 128
    (33, 144, 24, 16, 9, 1, False),      # two token tiles, and few weights
    (33, 1008, 64, 16, 49, 1, True), (64, 1040, 60, 16, 40, 2, True),      # weights just many enough to be streamed ..
    (49, 1008, 64, 16, 48, 1, False), (65, 1040, 60, 16, 40, 2, False),    # .. and just too few; a row too many
])
def test_few_token_layer_at_tile_edges(cb, tokens, d_model, blocks, block, active, stacked, streamed):
    from tests import harness as hz

    cfg = wl.FFNConfig("stream-edges", tokens, d_model, blocks * block, block, 16, stacked == 2, active / blocks, "uniform",
                       "normal", "normal0.02", stacked=stacked)
    r = hz.run_and_compare_products(cfg, seed=700 + tokens)
    assert r["mismatches"] == 0 and r["path"] == 2 and r["n_active"] == active * block, r
    assert r["kernels"] == [cb.KERNEL_STREAM if streamed else cb.KERNEL_LIMB] * 2


@pytest.mark.parametrize("tokens,d,n", [
    (16, 256, 96), (33, 1008, 784),                  # tiles of 32 features both ways; of 128
    (17, 1184, 128), (17, 1200, 128),                # 37 x 4 steps and 4 x 37; 38 x 4 and 4 x 38
    (32, 32, 2368), (32, 64, 2368),                  # 74 tiles of one step; of two, and 2 x 74
])
def test_tiles_of_a_few_token_layer(cb, tokens, d, n):
    """The multiply-adds that the statistics report are those of the tiles that ran: 32 features where every step of such tiles has an SM."""
    ctx = cb.Comet(tokens, d, n, 16, 12, max_active=n)
    assert ctx.set_mask(np.ones(n // 16, np.uint8)) == n
    shapes = {cb.W1: (n, d), cb.W2: (d, n), cb.X: (tokens, d), cb.A_UP: (tokens, d), cb.B_UP: (n, d), cb.C_UP: (tokens, n),
              cb.H: (tokens, n), cb.A_DN: (tokens, n), cb.B_DN: (d, n), cb.C_DN: (tokens, d)}
    zeros = {t: torch.zeros(s, dtype=torch.int64, device="cuda") for t, s in shapes.items()}
    for t, v in zeros.items():
        for p in (0, 1):
            ctx.bind_shares(p, t, v)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    up_to = lambda a, b: -(-a // b)  # noqa: E731
    for call, N, K in ((ctx.ffn_up, n, d), (ctx.ffn_down, d, n)):
        call(tokens)
        st = ctx.stats()
        steps = up_to(tokens, 32) * up_to(K, 32)
        features = 32 if steps * up_to(N, 32) <= sms else 128
        assert st.product_kernel == cb.KERNEL_STREAM
        assert st.tensor_tile_macs == 2 * 2 * steps * up_to(N, features) * features * 32 * 32, (N, K, features)
    ctx.synchronize()
    ctx.close()
