"""The binding's packed hom_problem and hom_inclusion records hold, member by member, what the
problem's description says."""
import ctypes
import shutil

import numpy as np
import pytest

import microstructures as ms

A3 = np.array([[2.0, 0.3, 0.1], [0.3, 1.0, -0.2], [0.1, -0.2, 1.5]])


@pytest.fixture(scope="module")
def bd():
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    import __graft_entry__
    __graft_entry__._builder().build()
    import paper_1404_3614_gb300.binding as bd
    return bd


PROBLEMS = {
    "homogeneous2d": lambda: ms.homogeneous(2, 5, np.array([[2.0, 0.3], [0.3, 1.0]])),
    "rect2d": lambda: ms.random_rectangles_2d(3, N=23),
    "aniso2d": lambda: ms.random_anisotropic_2d(1, N=7),
    "mixed3d": lambda: ms.make_problem(3, (9, 11, 13), (1.0, 0.8, 1.2), A3, [ms.ball((0.1, 0.0, 0.05), 0.3, 30.0, 3),
                                                                             ms.box((-0.3, 0.25, -0.4), (0.2, 0.1, 0.3), A3, 3)]),
}


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_packed_problem_holds_the_description(bd, name):
    pr = PROBLEMS[name]()
    d = pr.d
    p, keep = bd.problem_struct(pr)

    def padded(v, n, fill):
        return [float(x) for x in v] + [fill] * (3 - n)

    def block(A):
        M = np.zeros((3, 3))
        M[:d, :d] = A
        return list(M.reshape(-1))

    assert p.d == d and list(p.N) == [int(v) for v in padded(pr.N, d, 1)] and list(p.Y) == padded(pr.Y, d, 1.0)
    assert list(p.A0) == block(pr.A0) and p.n_incl == len(pr.inclusions)
    assert not p.bitmap and list(p.bitmap_n) == [1, 1, 1]
    assert p.closed == int(getattr(pr, "closed", False)) and p.smooth == int(getattr(pr, "smooth", False))
    for i, inc in enumerate(pr.inclusions):
        s = p.incl[i]
        assert s.shape == (bd.HOM_BOX if inc.shape == "box" else bd.HOM_BALL)
        assert list(s.center) == padded(inc.center, d, 0.0)
        assert list(s.size) == padded(inc.size, len(inc.size), 0.0)
        assert list(s.A) == block(inc.A)
    copy = (bd.hom_problem * 1)()
    copy[0] = p
    assert bytes(copy[0]) == bytes(p) and ctypes.sizeof(p) == bd._PROBLEM.size


def test_one_value_fills_every_axis(bd):
    """Counts, lengths and tensors given as one value or as lists, and a bitmap."""
    class P:
        d, N, Y, A0, inclusions, closed = 2, 7, 1, 1.5, [], True
        bitmap = np.arange(6.0).reshape(2, 3)
    p, keep = bd.problem_struct(P)
    assert list(p.N) == [7, 7, 1] and list(p.Y) == [1.0, 1.0, 1.0] and p.closed == 1
    assert list(p.A0)[:5] == [1.5, 1.5, 0.0, 1.5, 1.5]
    assert list(p.bitmap_n) == [2, 3, 1] and p.bitmap[:6] == [0.0, 3.0, 1.0, 4.0, 2.0, 5.0]
