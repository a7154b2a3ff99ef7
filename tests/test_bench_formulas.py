"""The counting rules behind the benchmark's throughput and roofline figures (CPU)."""
import importlib.util
import os

from paper_2505_07239_b200 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_algorithmic_macs_and_bytes_of_the_headline_configuration():
    b = _bench()
    cfg = wl.CONFIGS["opt1.3b"]
    n = cfg.n_active_blocks(0.9) * cfg.block
    assert n == 832
    T, d = cfg.tokens, cfg.d_model
    # 2 T K N per party per product, both parties, both projections
    assert b.ffn_macs(cfg, T, n) == 2 * 2 * T * d * n + 2 * 2 * T * n * d == 6_979_321_856
    # 8 (6 K N + 6 T K + 2 T N) bytes per party per product
    up = 8 * (6 * d * n + 6 * T * d + 2 * T * n)
    dn = 8 * (6 * n * d + 6 * T * n + 2 * T * d)
    assert b.ffn_bytes(cfg, T, n) == 2 * (up + dn) == 515_899_392


def test_gated_configuration_counts_both_stacked_matrices():
    b = _bench()
    cfg = wl.CONFIGS["llama7b"]
    n = 26 * cfg.block
    T, d = cfg.tokens, cfg.d_model
    assert cfg.groups == 2
    assert b.ffn_macs(cfg, T, n) == 2 * (2 * T * d * 2 * n) + 2 * (2 * T * n * d)


def test_workload_name_states_the_shape():
    b = _bench()
    name = b.workload_name(wl.CONFIGS["opt1.3b"], 0.9)
    for piece in ("tokens=512", "d_model=2048", "d_ff=8192", "sparsity=0.90", "n_active=832"):
        assert piece in name


def test_stored_traffic_is_keyed_by_the_kernel_source(monkeypatch):
    b = _bench()
    stored = b.COMBINE_LIMB_TRAFFIC
    workload, sparsity = stored["workload"]
    monkeypatch.setitem(stored, "kernel_sha256", b.combine_kernel_digest())       # the source is found
    assert b.combine_traffic(workload, sparsity, "combine_limb") == stored["bytes_per_launch"]
    assert b.combine_traffic(workload, sparsity, "combine_stream") is None
    assert b.combine_traffic("tiny", sparsity, "combine_limb") is None
    monkeypatch.setitem(stored, "kernel_sha256", "0" * 64)                        # another kernel than the profiled one
    assert b.combine_traffic(workload, sparsity, "combine_limb") is None
    # Planes once and Z read and written once.  Writes still in L2 at the kernel's end are not in the count, at this size all
    # of Z, 16 bytes a result word: what is left is read from memory, as every pass begins with an empty L2.
    cfg = wl.CONFIGS[workload]
    n, T, d = cfg.n_active_blocks(sparsity) * cfg.block, cfg.tokens, cfg.d_model
    once = 4 * ((3 * T * d + 3 * d * n + 4 * T * n) + (3 * T * n + 3 * n * d + 4 * T * d))
    assert once - 8 * (T * n + T * d) < stored["bytes_per_launch"] < 1.5 * once


def test_stored_traffic_of_the_residue_kernels():
    b = _bench()
    stored = b.COMBINE_RESIDUE_TRAFFIC
    workload, sparsity = stored["workload"]
    assert b.combine_kernel_digest("combine_residue") != b.combine_kernel_digest()
    assert b.combine_traffic(workload, sparsity, "combine_residue") in (None, stored["bytes_per_launch"])
    assert b.combine_traffic(workload, 0.5, "combine_residue") is None
    cfg = wl.CONFIGS[workload]
    n, T, d = cfg.n_active_blocks(sparsity) * cfg.block, cfg.tokens, cfg.d_model
    once = (b.product_bytes("combine_residue", T, d, n) + b.product_bytes("combine_residue", T, n, d)) // 2
    # all but the planes (51 bytes an operand word) and C (16 a result word) may stay in L2
    at_least = (51 * (T * d + T * n + 2 * n * d) + 16 * (T * n + T * d)) // 2
    assert at_least < stored["bytes_per_launch"] < 1.5 * once


def test_a_digest_is_that_of_the_code(tmp_path, monkeypatch):
    """Comments and white space aside, and over every file that the kernel is made of."""
    b = _bench()
    csrc = tmp_path / "paper_2505_07239_b200" / "csrc"
    csrc.mkdir(parents=True)
    texts = {}
    for source, _ in b.COMBINE_SOURCES["combine_residue"]:
        with open(os.path.join(ROOT, "paper_2505_07239_b200", "csrc", source)) as fh:
            texts[source] = fh.read()
    want = b.combine_kernel_digest("combine_residue")
    monkeypatch.setattr(b, "ROOT", str(tmp_path))

    def digest(**changed):
        for source, text in texts.items():
            (csrc / source).write_text(changed.get(source.split(".")[0], text))
        return b.combine_kernel_digest("combine_residue")

    assert digest() == want
    assert digest(kernels_residue=texts["kernels_residue.cuh"] + "\n// a comment more\n") == want
    assert digest(kernels_residue=texts["kernels_residue.cuh"] + "\nint x;\n") != want
    assert digest(residue_planes=texts["residue_planes.cuh"].replace("KC = 64", "KC = 32")) != want


def test_roofline_of_two_products_through_different_kernels():
    """The gated prompt: up through residues, down through limbs.  Each at the pipe's rate over its own byte products."""
    b = _bench()
    T, d, n = 256, 4096, 1664
    up, down = ("combine_residue", T, d, 2 * n), ("combine_limb", T, n, d)
    pipe, hbm = 60e12, 6450.0
    roof, macs = b.combine_roofline([up, down], 0.3, pipe, hbm)
    m_up, m_down = 4 * T * d * 2 * n, 4 * T * n * d
    seconds = m_up * 18 / 36 / pipe + m_down / pipe
    assert abs(macs * 1e12 / ((m_up + m_down) / seconds) - 1) < 1e-12
    assert roof["bound"] == "tensor" and abs(roof["frac"] / (seconds / 0.3e-3) - 1) < 1e-12
    assert roof["algorithmic_bytes_per_launch"] == (51 * (T * d + d * 2 * n) + 104 * T * 2 * n + 24 * (T * n + n * d) + 32 * T * d) // 2
    # a product whose bytes take longer than its multiply-adds is bound by them, whatever its kernel
    shallow = ("combine_residue", 512, 64, 8192)
    roof, _ = b.combine_roofline([shallow], 0.1, pipe, hbm)
    assert roof["bound"] == "hbm" and roof["unit"] == "GB/s"
    assert abs(roof["frac"] - b.product_bytes(*shallow) / (hbm * 1e9) / 1e-4) < 1e-9
