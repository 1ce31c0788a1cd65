"""The hr_lattice that a Lattice's calls pass: it follows bc and theta however they
are changed, and belongs to no caller."""

import ctypes
import pickle

import numpy as np
import pytest

from paper_2411_18511_gb300 import hr


@pytest.fixture
def passed(monkeypatch):
    """theta and bc as a call hands them to the library."""
    seen = []

    class Lib:
        def hr_gauge_packed_bytes(self, lat, rep, prec):
            seen.append((list(lat.dims), lat.bc, list(lat.theta)))
            return 0

    monkeypatch.setattr(hr, "lib", lambda: Lib())

    def call(lat):
        hr.hr_gauge_packed_bytes(lat, hr.HR_FUND, hr.HR_F64)
        return seen[-1]

    return call


def test_changes_in_place_and_by_assignment(passed):
    L = hr.Lattice((4, 6, 8, 10), 1)
    assert passed(L) == ([4, 6, 8, 10], 1, [0.0] * 4)
    for make in (list, np.array):
        L.theta = make([0.1, 0.0, 0.0, 0.2])
        assert passed(L)[2] == [0.1, 0.0, 0.0, 0.2]
        L.theta[0] = 0.7
        assert passed(L)[2] == [0.7, 0.0, 0.0, 0.2]
        L.theta = make([0.3, 0.0, 0.5, 0.0])  # a second array of the same kind
        assert passed(L)[2] == [0.3, 0.0, 0.5, 0.0]
    L.bc = 4
    assert passed(L)[1] == 4
    L.theta = None
    assert passed(L) == ([4, 6, 8, 10], 4, [0.0] * 4)
    assert passed(pickle.loads(pickle.dumps(L)))[0] == [4, 6, 8, 10]


def test_the_struct_of_lattice_is_the_callers_own(passed):
    L = hr.Lattice((4, 4, 4, 4), 0, (0.1, 0, 0, 0))
    passed(L)
    mine = hr.lattice(L)
    mine.bc, mine.theta[0], mine.dims[0] = 3, 9.0, 2
    assert passed(L) == ([4, 4, 4, 4], 0, [0.1, 0.0, 0.0, 0.0])
    assert hr.lattice(L).bc == 0 and ctypes.addressof(hr.lattice(L)) != ctypes.addressof(mine)


def test_extents_without_boundary_conditions(passed):
    assert passed((4, 4, 4, 6)) == ([4, 4, 4, 6], 0, [0.0] * 4)
