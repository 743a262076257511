"""The stage shapes and kernel names that the benchmark reports, against the library's sources (no GPU)."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2407_05568_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _shapes(text, launcher):
    """The shapes of a switch over P.tile in order: case 1 .. 4, with the default first."""
    cases = re.findall(r"(?:case (\d)|default): return " + launcher + r"<(?:2, )?(\d+), (\d+), (\d+)", text)
    found = [(int(k) if k else 0, (int(x), int(y), int(t))) for k, x, y, t in cases]
    return found


@pytest.mark.parametrize("precision,n,tile,shape,kernel", [
    ("fp64", (200,), 1, (8, 1, 128), "stage_line_fp64"), ("fp64", (2432,), 1, (8, 1, 128), "stage_line_fp64"),
    ("fp64", (2433,), 1, (62, 1, 128), "stage_kernel_fp64"), ("fp64", (65537,), 1, (254, 1, 256), "stage_kernel_fp64"),
    ("fp64", (128, 128), 1, (8, 8, 128), "stage_kernel_fp64"), ("fp64", (200, 200), 2, (25, 11, 384), "stage_kernel_fp64"),
    ("mixed", (200,), 1, (58, 1, 256), "stage_kernel_mixed1"), ("mixed", (17633,), 1, (254, 1, 256), "stage_kernel_mixed1"),
    ("mixed", (64, 64), 4, (20, 14, 608), "stage_kernel_mixed2")])
def test_reported_shapes(precision, n, tile, shape, kernel):
    got, name = bench.stage_shape(precision, n, tile, 152)
    assert got == shape and name.split("<")[0] == kernel
    assert re.search(r"\b" + kernel + r"\(StageParams", _source("es_stage.cu") + _source("es_stage_mixed.cu"))


def test_tables_are_the_sources():
    fp64 = _shapes(_source("es_stage.cu"), "launch_tile")
    small, large = dict(fp64[:5]), dict(fp64[5:])
    mixed = dict(_shapes(_source("es_stage_mixed.cu"), "launch_tile_f"))
    for table, name in ((small, "fp64 small"), (large, "fp64"), (mixed, "mixed")):
        assert {k + 1: v for k, v in table.items()} == bench.TILES[name]


def test_captured_kernels_exist():
    for name in bench.TRAFFIC_200:
        assert re.search(r"\b" + name.split("<")[0] + r"\b", _source("es_stage.cu") + _source("es_stage_mixed.cu"))
