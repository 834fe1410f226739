"""The bench's cited profile covers the files that hold the profiled kernel (no GPU)."""
import hashlib
import os

import bench

CSRC = os.path.join(bench.ROOT, "paper_2302_00414_gb300", "csrc")


def test_edit_of_any_named_source_retires_the_summary(tmp_path, monkeypatch):
    """Every file of the summary's `sources:` line is in the hash."""
    files = ["spread2d.cuh", "spreadmma.cuh", "common.cuh"]
    csrc = tmp_path / "paper_2302_00414_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for f in files + ["jobset.cuh"]:
        (csrc / f).write_text("// " + f + "\n")
    h = hashlib.sha256()
    for f in files:
        h.update((csrc / f).read_bytes())
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "s.md").write_text(
        f"kernel: k\nsources: {' '.join(files)}\nsource_sha256: {h.hexdigest()[:16]}\n"
        "dram_bytes_per_launch: 7\nsmem_pipe_frac: 0.5\nissue_frac: 0.6\ntensor_frac: 0.25\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    whole = {"dram_bytes_per_launch": 7.0, "smem_pipe_frac": 0.5, "issue_frac": 0.6, "tensor_frac": 0.25}
    assert bench.profiled("s.md", kernel="k") == whole
    for f in files:
        text = (csrc / f).read_text()
        (csrc / f).write_text(text + "// edited\n")
        assert bench.profiled("s.md", kernel="k") == {}
        (csrc / f).write_text(text)
    assert bench.profiled("s.md", kernel="k") == whole


def test_committed_summary_names_the_file_of_the_kernel_body():
    text = open(os.path.join(bench.ROOT, "profiles", "k_spread2d_batched_d2_m4.md")).read()
    sources = [ln for ln in text.splitlines() if ln.startswith("sources:")][0].split()[1:]
    assert "spreadmma.cuh" in sources and "spread2d.cuh" in sources
    assert "spread2d_mma_item" in open(os.path.join(CSRC, "spreadmma.cuh")).read()
