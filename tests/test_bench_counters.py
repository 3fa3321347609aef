"""Profiler figures in the bench line: of a kernel whose code is no longer the captured one there are none."""
import json
import os

import bench


def counters(tmp_path, monkeypatch, digests):
    with open(os.path.join(bench.ROOT, "profiles", "ncu_counters.json")) as f:
        captured = json.load(f)
    captured["source_digests"] = digests
    os.makedirs(tmp_path / "profiles")
    (tmp_path / "profiles" / "ncu_counters.json").write_text(json.dumps(captured))
    os.symlink(os.path.join(bench.ROOT, "paper_2601_02311_b200"), tmp_path / "paper_2601_02311_b200")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return {k for w in bench.ncu_counters()["workloads"].values() for k in w["kernels"]}


def test_figures_of_other_code_are_left_out(tmp_path, monkeypatch):
    got = counters(tmp_path, monkeypatch, {"k_sweep": "of other code", "k_eval": bench.source_digest("k_eval")})
    assert got == {"k_eval_materialise"}


def test_figures_of_this_code_are_given(tmp_path, monkeypatch):
    got = counters(tmp_path, monkeypatch, {k: bench.source_digest(k) for k in bench.KERNEL_SOURCES})
    assert got == {"k_sweep_topk", "k_sweep_pareto", "k_eval_materialise"}


def test_a_capture_that_does_not_name_its_code_gives_none(tmp_path, monkeypatch):
    assert counters(tmp_path, monkeypatch, {}) == set()


def test_comments_and_spacing_do_not_count(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2601_02311_b200" / "csrc"
    os.makedirs(csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    seen = []
    for sweep in ("int a; // one\n", "/* two\n */ int  a;", "int b;"):
        for name in ("ps_sweep.cu",) + bench.HEADERS:
            (csrc / name).write_text(sweep if name == "ps_sweep.cu" else "")
        seen.append(bench.source_digest("k_sweep"))
    assert seen[0] == seen[1] != seen[2]
