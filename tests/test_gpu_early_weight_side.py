"""Where ffn_up opens the weight side of the down-projection: in the launch of its own exchange, or in a launch beside its product, which
is one launch more.  The rule goes by that side's words and by the multiply-adds of the product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _launches(cb, tokens, d, blocks, clusters, early):
    """Launches of one ffn_up on zeros, with or without the down-projection's triple there already."""
    n = 16 * blocks
    stream = torch.cuda.Stream()
    ctx = cb.Comet(tokens, d, n, 16, 12, max_active=n, stream=stream)
    shapes = {cb.W1: (n, d), cb.W2: (d, n), cb.X: (tokens, d), cb.A_UP: (tokens, d), cb.B_UP: (n, d), cb.C_UP: (tokens, n)}
    if early:
        shapes.update({cb.B_DN: (d, n), cb.C_DN: (tokens, d)})
    zeros = {t: torch.zeros(s, dtype=torch.int64, device="cuda") for t, s in shapes.items()}
    torch.cuda.synchronize()
    ctx.set_mask(np.ones(blocks, np.uint8))
    if clusters:                                 # tokens and blocks in as many equal groups, every block used by its group
        group = lambda count: np.arange(count) * clusters // count  # noqa: E731
        ctx.set_token_mask((group(tokens)[:, None] == group(blocks)[None, :]).astype(np.uint8))
    for t, v in zeros.items():
        for p in (0, 1):
            ctx.bind_shares(p, t, v)
    before = ctx.stats().kernel_launches
    ctx.ffn_up(tokens)
    after = ctx.stats()
    ctx.synchronize()
    ctx.close()
    assert after.product_kernel == (cb.KERNEL_GROUPED if clusters else cb.KERNEL_LIMB)
    return after.kernel_launches - before


@pytest.mark.parametrize("tokens,d,blocks,clusters,apart", [
    (200, 864, 16, 0, False), (200, 960, 16, 0, True),        # 0.2 million words, 44 and 49 million multiply-adds
    (512, 512, 12, 0, False), (512, 512, 13, 0, True),        # 0.1 million words, 50 and 55 million
    (2048, 256, 15, 0, False), (2048, 256, 16, 0, True),      # 126 and 134 million, just fewer words than it takes and as many
    (400, 512, 32, 0, True),                                  # so many words that it takes no long product
    (512, 512, 12, 4, False), (512, 512, 16, 4, True),        # in groups the union's multiply-adds count
])
def test_launch_of_the_weight_side(tokens, d, blocks, clusters, apart):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding as cb

    late, early = (_launches(cb, tokens, d, blocks, clusters, e) for e in (False, True))
    assert early - late == apart
