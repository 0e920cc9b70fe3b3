"""The recorded DRAM traffic of the bench is that of the present kernels, and falls away when they change."""

import os
import shutil

import pytest

import bench


def _copy_of_sources(tmp_path):
    dst = tmp_path / "paper_2606_08883_gb300" / "csrc"
    shutil.copytree(os.path.join(bench.ROOT, "paper_2606_08883_gb300", "csrc"), dst)
    return dst


def test_every_record_is_of_the_present_kernels():
    assert bench.krylov_traffic(1 << 20, 10, 30) is not None
    for name, prec in bench.NCU_TRAFFIC:
        assert bench.ncu_traffic(name, prec) is not None, name


@pytest.mark.parametrize("changed", ["common.cuh", "k_local.cu", "k_krylov.cu"])
def test_a_changed_source_drops_the_record(tmp_path, monkeypatch, changed):
    src = _copy_of_sources(tmp_path)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.ncu_traffic("schwarz", "fp32") and bench.krylov_traffic(1 << 20, 10, 30)
    with open(src / changed, "a") as f:
        f.write("\n")
    assert (bench.ncu_traffic("schwarz", "fp32") is None) == (changed != "k_krylov.cu")
    assert (bench.krylov_traffic(1 << 20, 10, 30) is None) == (changed != "k_local.cu")
