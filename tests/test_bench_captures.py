"""The capture figures of bench.py's roofline block are those of the profile files that it names as their source."""
import os

import pytest

import bench

UNITS = {"byte": 1.0, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9, "%": 0.01}


def _table(path):
    out = {}
    with open(os.path.join(bench.ROOT, path)) as f:
        for line in f:
            cells = [c.strip() for c in line.split("|")]
            if len(cells) == 4 and "(`" in cells[1]:
                value, _, unit = cells[2].partition(" ")
                if unit in UNITS:
                    out[cells[1].split("(`")[1].rstrip("`)")] = float(value.replace(",", "")) * UNITS[unit]
    return out


@pytest.mark.parametrize("kernel", ["pm_sweep", "pm_sweep_plane"])
def test_captured_figures_are_those_of_the_named_file(kernel):
    traffic, source = bench.TRAFFIC_PER_LAUNCH[kernel]
    t = _table(source)
    assert traffic == pytest.approx(t["dram__bytes_read.sum"] + t["dram__bytes_write.sum"], rel=1e-6)
    issue, source = bench.ISSUE_PER_LAUNCH[kernel]
    assert issue == pytest.approx(_table(source)["smsp__issue_active.avg.pct_of_peak_sustained_active"], rel=1e-6)


def test_a_missing_figure_is_none(tmp_path):
    (tmp_path / "p.md").write_text("| write (`dram__bytes_write.sum`) | 1,024.5 Kbyte |\n| n (`x.sum`) | 3 inst |\n")
    path = str(tmp_path / "p.md")
    assert bench._captured(path, "dram__bytes_write.sum") == pytest.approx(1024500)
    assert bench._captured(path, "x.sum") == 3 and bench._captured(path, "dram__bytes_read.sum") is None
    assert bench._traffic(path) is None and bench._captured(str(tmp_path / "none.md"), "x.sum") is None
