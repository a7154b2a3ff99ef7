"""Both forms of the shuffle, one pass (matrices of up to 2^21 words, rows of one or two words up to fewer) and two, against the CPU oracle, bit for bit."""
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


# 2^21 words exactly; just above, in 16-byte and in 8-byte pieces; one row longer than the limit; both sides of the line for
# rows of one and of two words
@pytest.mark.parametrize("rows,cols", [(1024, 2048), (1025, 2050), (699, 3001), (1, (1 << 21) + 2),
                                       (148 << 10, 1), ((148 << 10) + 1, 1), (3 << 16, 2), ((3 << 16) + 1, 2)])
@pytest.mark.parametrize("bad", [False, True])
def test_shuffle_on_both_sides_of_the_limit(cb, rows, cols, bad):
    seed = 900 + rows
    x = wl.random_u64(seed, "x", rows * cols).reshape(rows, cols)
    xs = wl.split_shares(x, seed, "x")
    m = wl.dealer_shuffle(seed, "sh", rows, cols)
    rho = [r.copy() for r in m["rho"]]
    if bad:
        rho[1][rows // 2] = -3                       # never followed: the row counts as zero, and the flag is raised
    ref = [r.copy() for r in rho]
    ref[1][rows // 2] = m["rho"][1][rows // 2]
    y_ref, z_ref = oracle.shuffle_online(xs, m["tau"], ref, m["a"], m["b"])
    if bad:
        z_ref[1][rows // 2] = np.uint64(0) - m["b"][1][rows // 2]
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    d64 = lambda v: cb.to_device(v)  # noqa: E731
    d32 = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.int32)).cuda()  # noqa: E731
    Y, Z = cb.shuffle([d64(v) for v in xs], [d32(v) for v in m["tau"]], [d32(v) for v in rho], [d64(v) for v in m["a"]],
                      [d64(v) for v in m["b"]], bad_index_flag=flag)
    torch.cuda.synchronize()
    for i in (0, 1):
        assert np.array_equal(Y[i].cpu().numpy().view(np.uint64), y_ref[i]), i
        assert np.array_equal(Z[i].cpu().numpy().view(np.uint64), z_ref[i]), i
    assert int(flag.item()) == int(bad)
