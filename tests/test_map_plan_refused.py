"""Which graphs the spin-map engine's host plan refuses: exactly the ones whose
tables do not fit in a block's shared memory, of those that test_map_plan.py
walks. A plan that is refused for any other reason would leave its graph to a
slower engine, with the same spins."""

import subprocess

import pytest

from test_map_plan import BLOCK, BLOCK_STREAM, CLUSTER, COMPLETE, GRID, LONG_ROWS, PAIRS, check  # noqa: F401

FORMS = [(BLOCK, 1), (BLOCK_STREAM, 1), (CLUSTER, 2), (CLUSTER, 16), (GRID, 7), (GRID, 152)]
GRAPHS = [(PAIRS, 1, 0, 1), (PAIRS, 2, 1, 1), (PAIRS, 33, 40, 2), (PAIRS, 799, 19000, 1), (PAIRS, 4095, 20000, 30),
          (PAIRS, 20011, 300000, 8), (PAIRS, 199999, 400000, 1), (COMPLETE, 90, 0, 1), (LONG_ROWS, 9001, 21, 3)]
# one block with its entries in shared memory, and a map of 200,000 spins beside
# the tasks of anything but 152 blocks
REFUSED = {(799, BLOCK, 1, 1), (4095, BLOCK, 1, 0), (4095, BLOCK, 1, 1), (20011, BLOCK, 1, 0), (20011, BLOCK, 1, 1),
           (9001, BLOCK, 1, 1)} | {(199999, mode, K, wide) for mode, K in FORMS[:-1] for wide in (0, 1)}


@pytest.mark.parametrize("kind,n,m,wmax", GRAPHS)
def test_refused_plans(check, kind, n, m, wmax):  # noqa: F811
    for mode, K in FORMS:
        for wide in (0, 1):
            r = subprocess.run([check] + [str(x) for x in (kind, n, m, wmax, mode, K, wide, 7)], capture_output=True,
                               text=True)
            assert r.returncode == (2 if (n, mode, K, wide) in REFUSED else 0), (mode, K, wide, r.stdout)
