"""Which kernel segments a launch's problems (segment.cuh): a device that cannot
place the 16-CTA cluster gets the kernels that run anywhere, with the lines at
which one CTA and the grid meet there."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
WARP, CLUSTER, GRID, CTA = range(4)


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("route") / "segment_route")
    subprocess.run([cxx, "-std=c++17", os.path.join(HERE, "host", "segment_route.cpp"), "-o", exe],
                   check=True)

    def ask(*rows):
        text = "\n".join(" ".join(str(int(x)) for x in row) for row in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [int(x) for x in out.split()]

    return ask


def test_routes(route):
    one = [1, 32, 33, 4095, 4096, 8191, 8192, 81920, 81921, 1 << 30]
    assert route(*[(1, n, 1, 1) for n in one]) == [
        WARP, WARP, CTA, CTA, CLUSTER, CLUSTER, CLUSTER, CLUSTER, GRID, GRID]
    # no cluster on this device: one CTA up to 8191 tokens, the grid from there
    assert route(*[(1, n, 1, 0) for n in one]) == [
        WARP, WARP, CTA, CTA, CTA, CTA, GRID, GRID, GRID, GRID]
    # several problems, or no status word for a wait that gives up
    assert route(*[(p, n, s, f) for n in one for p, s in ((2, 1), (1, 0)) for f in (0, 1)]) == [
        WARP] * 8 + [CTA] * 32
