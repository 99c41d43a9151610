"""The circuits of test_support_cpu.py again, with a deviation that counts an amplitude that is
not a number (support_suite.cpp's maximum passes over it; circuit_suite.cpp's does not)."""
import numpy as np
import pytest

import test_support_cpu as circuits
from test_phase_runs import suite  # noqa: F401  (the suite that reports "nan")


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
@pytest.mark.parametrize("n,count", [(12, 40), (18, 24)])
def test_random_rotations(suite, tmp_path, n, count, dtype, tol):  # noqa: F811
    circuits.test_random_rotations(suite, tmp_path, n, count, dtype, tol)


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
@pytest.mark.parametrize("orbitals,masks", [(7, 70), (9, 60)])
def test_molecular_strings(suite, tmp_path, orbitals, masks, dtype, tol):  # noqa: F811
    circuits.test_molecular_strings(suite, tmp_path, orbitals, masks, dtype, tol)


def test_written_by_its_owner(suite, tmp_path):  # noqa: F811
    n = 18
    rots = circuits._random(n, 10, np.random.default_rng(3))
    status, worst, parts, _ = circuits._run(suite, tmp_path, n, rots, "c128")
    assert status == 0 and worst < 1e-12 and parts > 0
    # every pass that would have visited a part finds amplitudes elsewhere
    status, worst, parts, _ = circuits._run(suite, tmp_path, n, rots, "c128", ((1 << n) - 7,))
    assert status == 0 and worst < 1e-12 and parts == 0
