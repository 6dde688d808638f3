"""What voids the committed ncu record of the wavefronts: any change to the layout of the cells, to the
code that moves them or that updates loads, or to the launcher; not one to the kernels that build cells."""
import json
import os

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KERNEL = "k_sweep_systolic"


@pytest.fixture
def hash_of(monkeypatch, tmp_path):
    def f(text):
        d = tmp_path / "paper_2307_15969_gb300" / "csrc"
        d.mkdir(parents=True, exist_ok=True)
        (d / "systolic.cu").write_text(text)
        monkeypatch.setattr(bench, "ROOT", str(tmp_path))
        return bench._sweep_hash(KERNEL)
    return f


def test_spans(hash_of):
    src = open(os.path.join(ROOT, "paper_2307_15969_gb300", "csrc", "systolic.cu")).read()
    base = bench._sweep_hash(KERNEL)
    assert base != "missing"
    for inside in ("struct Geo {", "void fetch_chunk(", "void store_split(", "float transfer(", "void run_chunks(",
                   "void step_any(", "k_sweep_systolic(const SysArgs a) {", "cudaError_t lowd_sys_passes("):
        assert src.count(inside) == 1, inside
        i = src.index(inside) + len(inside)
        assert hash_of(src[:i] + " " + src[i:]) != base, inside
    for outside in ("void k_cells_from_edges(", "bool lowd_sys_serves("):
        i = src.index(outside) + len(outside)
        assert hash_of(src[:i] + " " + src[i:]) == base, outside


def test_record_is_of_the_current_source():
    with open(os.path.join(ROOT, "profiles", "k_sweep_systolic_rmat22_dram.json")) as f:
        d = json.load(f)
    assert d["sweep_cu_sha256_16"] == bench._sweep_hash(KERNEL)
    assert bench._traffic_per_pass(KERNEL) == float(d["dram_bytes_per_pass"])
