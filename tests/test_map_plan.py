"""The spin-map engine's host plan, walked on the CPU the way the kernel walks
it (map_plan_check.cpp): every index in bounds, every row decided once, every
flip word drawn once, and the spins of three sweeps equal to a plain sweep's."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_10750_gb300", "csrc")
PAIRS, COMPLETE, LONG_ROWS, HUBS = 0, 1, 2, 3
BLOCK, BLOCK_STREAM, CLUSTER, GRID = 0, 1, 2, 3


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("map") / "map_plan_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-pthread", "-o", exe,
                    os.path.join(ROOT, "tests", "map_plan_check.cpp"), os.path.join(CSRC, "host_graph.cpp"),
                    os.path.join(CSRC, "map_plan.cpp")], check=True)
    return exe


@pytest.mark.parametrize("kind,n,m,wmax", [
    (PAIRS, 1, 0, 1), (PAIRS, 2, 1, 1), (PAIRS, 33, 40, 2), (PAIRS, 799, 19000, 1), (PAIRS, 4095, 20000, 30),
    (PAIRS, 20011, 300000, 8), (PAIRS, 199999, 400000, 1), (COMPLETE, 90, 0, 1), (LONG_ROWS, 9001, 21, 3),
])
@pytest.mark.parametrize("mode,K", [(BLOCK, 1), (BLOCK_STREAM, 1), (CLUSTER, 2), (CLUSTER, 16), (GRID, 7),
                                    (GRID, 152)])
def test_plan_sweeps_like_the_rows(check, kind, n, m, wmax, mode, K):
    for wide in (0, 1):
        r = subprocess.run([check] + [str(x) for x in (kind, n, m, wmax, mode, K, wide, 7)], capture_output=True,
                           text=True)
        # 2: the tables do not fit (resident entries of a large graph, a map of
        # 200,000 spins beside too many tasks)
        assert r.returncode == 0 or (r.returncode == 2 and n * max(m, n) > 10 ** 6), r.stdout


@pytest.mark.parametrize("kind,n,m", [(HUBS, 4097, 1), (HUBS, 9001, 40), (HUBS, 30000, 300), (COMPLETE, 300, 0),
                                      (PAIRS, 5000, 4000)])
@pytest.mark.parametrize("K", [1, 8, 16])
def test_split_rows_sweep_like_the_rows(check, kind, n, m, K):
    for wide in (0, 1):
        r = subprocess.run([check] + [str(x) for x in (kind, n, m, 5, CLUSTER, K, wide, 3, 1)], capture_output=True,
                           text=True)
        # 2: the tables of 30,000 rows do not fit in one block, nor a map of 300 classes on 16
        assert r.returncode == (2 if (n, K) in ((30000, 1), (300, 16)) else 0), r.stdout


@pytest.mark.parametrize("K", [1, 2, 4, 8, 16])
def test_batch_tables(tmp_path, K):
    exe = str(tmp_path / "batch_map_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-pthread", "-o", exe,
                    os.path.join(ROOT, "tests", "batch_map_check.cpp"), os.path.join(CSRC, "host_graph.cpp"),
                    os.path.join(CSRC, "batch_map_plan.cpp")], check=True)
    r = subprocess.run([exe, str(K), "3"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
