"""The exchange kernel (messages and operand planes of the tensor-core path, more than 32 token rows) at the edges of its
tiles: 16 rows per CTA, k-blocks of 32 words, up to 16 k-blocks per CTA.  Bit for bit against the CPU oracle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2505_07239_b200 import workloads as wl  # noqa: E402


@pytest.mark.parametrize("early_down", [True, False])     # weight side of the down-projection beside the up-projection, or not
@pytest.mark.parametrize("tokens,d_model,blocks,block,active,stacked", [
    (33, 16, 4, 16, 1, 1),          # half a k-block deep both ways, one row beyond two CTAs
    (48, 560, 40, 16, 35, 1),       # 17.5 k-blocks: more than a CTA's share, a half block at the end
    (127, 96, 9, 48, 5, 2),         # strips of 48 columns: a k-block takes its halves from two blocks
    (257, 272, 6, 80, 3, 3),        # three stacked matrices, ragged row tiles
])
def test_layer_at_exchange_tile_edges(tokens, d_model, blocks, block, active, stacked, early_down):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from tests import harness as hz

    cfg = wl.FFNConfig("exchange-edges", tokens, d_model, blocks * block, block, 16, stacked == 2, active / blocks,
                       "uniform", "normal", "normal0.02", stacked=stacked)
    r = hz.run_and_compare_products(cfg, seed=800 + tokens, early_down=early_down)
    assert r["mismatches"] == 0 and r["path"] == 2 and r["n_active"] == active * block, r
