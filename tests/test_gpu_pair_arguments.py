"""The two parties' tensors as something other than a list: one stacked tensor, and a sequence that makes its items when asked.
Every entry point that takes pairs gives the same words as with lists."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class _OnDemand:
    """Items are copies that nobody else holds."""

    def __init__(self, stacked):
        self.stacked = stacked

    def __getitem__(self, i):
        return self.stacked[i].clone()


def _as(form, stacked):
    return {"list": lambda: [stacked[0].clone(), stacked[1].clone()], "stacked": stacked.clone,
            "on demand": lambda: _OnDemand(stacked)}[form]()


@pytest.mark.parametrize("form", ["stacked", "on demand"])
def test_pairs_in_every_form(form):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_07239_b200 import binding as cb

    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)

    def words(*shape):
        return torch.randint(-(1 << 63), (1 << 63) - 1, (2, *shape), dtype=torch.int64, device="cuda", generator=gen)

    rows, cols, T, K, N = 40, 24, 5, 24, 40
    x, y, a, b, c = (words(rows, cols) for _ in range(5))
    perm = [torch.stack([torch.randperm(rows, device="cuda", generator=gen) for _ in (0, 1)]).int() for _ in (0, 1)]
    X, A, Y, B, C = words(T, K), words(T, K), words(N, K), words(N, K), words(T, N)

    def calls(f):
        out = [*cb.shuffle(_as(f, x), _as(f, perm[0]), _as(f, perm[1]), _as(f, a), _as(f, b)),
               *cb.beaver_mul(_as(f, x), _as(f, y), _as(f, a), _as(f, b), _as(f, c))]
        # written in place: a sequence that makes copies keeps nothing of that, so the written operand is none here
        z = _as("list" if f == "on demand" else f, x)
        out.append(cb.truncate_pair(z, _as(f, a), _as(f, b), 12))
        cb.add_bias(z, _as(f, c[:, 0].contiguous()))
        out.append(z)
        Z = torch.zeros((2, T, N), dtype=torch.int64, device="cuda")
        assert cb.beaver_matmul_static(_as(f, X), _as(f, A), _as(f, Y), _as(f, B), _as(f, C), [Z[0], Z[1]]) == cb.OK
        out.append(Z)
        torch.cuda.synchronize()
        return out

    for got, want in zip(calls(form), calls("list"), strict=True):
        for p in (0, 1):
            assert torch.equal(got[p], want[p])
