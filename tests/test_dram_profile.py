"""The committed DRAM bytes of the 1024^3 / 2048^3 kernels that exist now: the table's algorithmic bytes
are those bench.py credits, no launch moved less, and the traffic file holds the table's figures."""
import json
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N_P, NG = 1024, 2048


def rows():
    """label -> (kernel, read GB, write GB, algorithmic GB)"""
    text = open(os.path.join(ROOT, "profiles", "dram_cola_1024p_2048g.md")).read()
    out = {}
    for m in re.finditer(r"^\| `([^`]+)` \| (\w+) \| [\d.]+ \| ([\d.]+) \| ([\d.]+) \| \d+ \| [\d.]+ \| ([\d.]+) \|", text, re.M):
        out[m.group(2)] = (m.group(1), *(float(m.group(i)) for i in (3, 4, 5)))
    return out


def test_table_names_kernels_of_the_sources():
    csrc = os.path.join(ROOT, "paper_1301_0322_gb300", "csrc")
    source = "".join(open(os.path.join(csrc, f)).read() for f in os.listdir(csrc))
    assert len(rows()) == 9
    for kernel, *_ in rows().values():
        assert re.search(r"\b%s\(" % kernel.split("<")[0], source), kernel


def test_table_agrees_with_the_bench_and_the_traffic_file():
    traffic = json.load(open(os.path.join(ROOT, "profiles", "ncu_traffic_1024p_2048g.json")))["cola_1024p_2048g_L1000"]
    for label, (kernel, rd, wr, alg_gb) in rows().items():
        alg = bench.algorithmic_bytes(label, N_P, NG)
        assert abs(alg / 1e9 - alg_gb) <= 0.006, label
        assert (rd + wr) * 1e9 >= 0.99 * alg, label
        rec = traffic[label.replace("fft_cols_", "fft_cols_fwd_")]
        assert abs(rec["dram_bytes_per_launch"] / 1e9 - (rd + wr)) <= 0.011, label


def test_bench_reports_traffic_of_the_digest_it_was_taken_on(monkeypatch):
    rec = json.load(open(os.path.join(ROOT, "profiles", "ncu_traffic_1024p_2048g.json")))["cola_1024p_2048g_L1000"]
    monkeypatch.setattr(bench, "kernel_source_digest", lambda: rec["fft_z_green_2048"]["source_digest"])
    got = bench.measured_traffic("fft_z_green_2048", "cola_1024p_2048g_L1000")
    assert got == rec["fft_z_green_2048"]["dram_bytes_per_launch"]
    monkeypatch.setattr(bench, "kernel_source_digest", lambda: "another")
    assert bench.measured_traffic("fft_z_green_2048", "cola_1024p_2048g_L1000") is None
