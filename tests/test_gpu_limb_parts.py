"""The limb kernel's two ways to cut its work, at the lines between them: equal ranges of all tiles' blocks, and every tile in parts of
its own.  Tiles are 128 x 64 words, blocks 32 contraction indices; both products of a layer, bit for bit against the CPU oracle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2505_07239_b200 import workloads as wl  # noqa: E402


@pytest.mark.parametrize("tokens,d_model,active", [
    (33, 48, 1),           # 2 tiles of 4 blocks: no more blocks than SMs, ranges of one
    (128, 304, 28),        # 14 tiles of 20 blocks in 10 parts; 10 of 28 in 14
    (129, 208, 44),        # two token tiles, the second with one row: 44 tiles of 14 blocks in 3 parts of 4 and 5
    (260, 64, 52),         # 78 tiles of 4 blocks, a part each; 6 of 52 blocks in 18 parts
    (260, 64, 101),        # 156 tiles: more than SMs, ranges
    (97, 1040, 8),         # 4 tiles of 66 blocks in 33 parts; 34 tiles of 8 blocks in 4
    (200, 960, 16), (200, 864, 16),      # the down-projection's weight side opened beside the product, and in the launch before it
])
def test_layer_in_parts(tokens, d_model, active):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding as cb
    from tests import harness as hz

    cfg = wl.FFNConfig("limb-parts", tokens, d_model, (active + 3) * 16, 16, 16, False, active / (active + 3), "uniform", "normal",
                       "normal0.02", stacked=1)
    r = hz.run_and_compare_products(cfg, seed=600 + tokens)
    assert r["mismatches"] == 0 and r["n_active"] == active * 16, r
    assert r["kernels"] == [cb.KERNEL_LIMB] * 2
