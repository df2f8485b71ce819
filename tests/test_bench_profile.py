"""The DRAM traffic that the benchmark reports belongs to the counting kernels
as they are: the committed capture names their code, comments and blanks aside."""
import re

import bench


def test_profile_is_of_the_current_kernels():
    assert bench.profiled_traffic(1 << 40) is not None
    # scaled by the ratio of algorithmic bytes, 1 on the captured graph
    text = open(bench.os.path.join(bench.ROOT, "profiles", "counting_kernels_rmat_s24.txt")).read()
    kv = dict(re.findall(r"^(\w+): (\d+)$", text, re.M))
    total = int(kv["dram_bytes_per_launch"])
    assert bench.profiled_traffic(int(kv["algorithmic_bytes_per_launch"])) == total
    assert total == sum(int(kv[f"{k}_dram_bytes_{d}"]) for k in ("k_tri_hub", "k_triangles")
                        for d in ("read", "write"))


def test_a_change_of_code_is_noticed(tmp_path, monkeypatch):
    src = open(bench.os.path.join(bench.ROOT, "paper_2012_11188_gb300", "csrc", "triangles.cu")).read()
    csrc = tmp_path / "paper_2012_11188_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").symlink_to(bench.os.path.join(bench.ROOT, "profiles"))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (csrc / "triangles.cu").write_text("// another comment\n" + src.replace("  ", "    "))
    assert bench.profiled_traffic(1 << 40) is not None
    (csrc / "triangles.cu").write_text(src.replace("constexpr int HUB_PAIRS = 4;",
                                                   "constexpr int HUB_PAIRS = 5;"))
    assert bench.profiled_traffic(1 << 40) is None
