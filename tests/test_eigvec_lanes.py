"""The warp form of the eigenvectors of T (tridiag_vec.cuh) on the CPU, its 32
lanes run one after the other between their meeting points: a lane must not
read an entry that another lane may already have overwritten, whatever the
order in which the lanes run."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2607_19368_gb300 import build
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))),
                           "include")
    exe = str(tmp_path_factory.mktemp("eigvec") / "eigvec_lanes")
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I", include,
                    os.path.join(HERE, "host", "eigvec_lanes.cpp"), "-o", exe], check=True)
    return exe


def matrices():
    g = np.random.default_rng(3)
    out = {"one": (np.array([2.0]), np.zeros(1)), "two": (np.array([1.0, 3.0]), np.array([0.5, 0]))}
    for n in (5, 16, 31, 32, 33, 64, 100, 128):
        a, b = 1.0 + g.random(n), 0.5 * g.random(n)
        out[f"random {n}"] = (a, b)
    n = 33  # Ritz values of a feature matrix: falling over many decades
    s = 10.0 ** -np.linspace(0, 8, n)
    out["graded"] = (s, 0.3 * np.sqrt(s * np.append(s[1:], 0.0)))
    w = np.abs(np.arange(-10, 11)).astype(float) + 1.0  # Wilkinson: pairs of close values
    out["wilkinson"] = (w, np.ones(21))
    return out


@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(matrices()))
def test_eigenvectors_do_not_depend_on_lane_order(program, name, order):
    a, b = matrices()[name]
    n = a.size
    T = np.diag(a) + np.diag(b[:n - 1], 1) + np.diag(b[:n - 1], -1)
    th = np.linalg.eigvalsh(T)[::-1].copy()
    text = " ".join([str(order), str(n)] + [float(x).hex() for x in np.concatenate([a, b, th])])
    out = subprocess.run([program], input=text, capture_output=True, text=True, check=True).stdout
    S = np.array([[float.fromhex(x) for x in row.split()] for row in out.splitlines()])
    # double-float solves: 2^-44 |T| per shift over gaps of at least 1e-7 |T| outside a
    # cluster, products of n terms
    assert np.abs(S.T @ S - np.eye(n)).max() <= n * 2.0 ** -44 / 1e-7
    assert np.abs(T @ S - S * th).max() <= 16 * n * 2.0 ** -44 * np.abs(th).max()
