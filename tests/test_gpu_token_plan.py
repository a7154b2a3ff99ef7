"""The components a per-token mask falls into (comet_set_token_mask's plan) at the edges of what the kernel distinguishes:
rows in 32s and the first 64, block words of 32, masks off a 16-byte boundary, working storage in and out of shared memory,
more tokens than the sorted order covers, and a chain that joins every block to the next.  Against the oracle's search."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402


def _labels(comp):
    """Component numbers -> the smallest token index of the component, -1 for none."""
    first = {}
    for r, c in enumerate(comp[0].tolist()):
        first.setdefault(c, r)
    first[-1] = -1
    return [np.array([first[c] for c in part.tolist()], np.int64) for part in comp]


@pytest.mark.parametrize("T,nab,density,shift", [
    (1, 1, 1.0, 0), (33, 1, 0.5, 0), (64, 32, 0.02, 0), (65, 31, 0.03, 4), (500, 33, 0.004, 1), (517, 26, 0.003, 0),
    (129, 128, "chain", 0), (130, 200, "chain", 8),
    (4100, 70, 0.0004, 0),        # 12300 words of bits: working storage in global memory
    (33000, 16, 0.00003, 0),      # labels and counts alone
    (300, 40, 0.0, 0),            # no edge at all
])
def test_components_of_a_token_mask(T, nab, density, shift):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding as cb

    if density == "chain":                               # token r uses blocks r and r + 1, tokens in shuffled order
        S = np.zeros((T, nab), np.uint8)
        for r, t in enumerate(np.random.default_rng(5).permutation(T).tolist()):
            S[t, [min(r, nab - 1), min(r + 1, nab - 1)]] = 1
    else:
        S = (np.random.default_rng(T + nab).random((T, nab)) < density).astype(np.uint8)
    rows, cols, n = oracle.components_dfs(S)
    want_rows, want_cols = _labels((rows, cols))
    ctx = cb.Comet(T, 16, 16 * nab, 16, 12, 0)
    ctx.set_mask(np.ones(nab, np.uint8))
    buffer = torch.zeros(T * nab + shift, dtype=torch.uint8, device="cuda")
    on_device = buffer[shift:].view(T, nab)              # starts `shift` bytes off a 256-byte boundary
    on_device.copy_(torch.from_numpy(S))
    for mask in (on_device, S):
        assert ctx.set_token_mask(mask) == 16 * int(S.sum())
        row_label, blk_label, count = ctx.get_components(T, nab)
        assert count == n and np.array_equal(row_label, want_rows) and np.array_equal(blk_label, want_cols)
    ctx.close()
