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


class Description:
    """A problem of one size in every direction; members replaced by keyword."""
    def __init__(self, d, **kw):
        self.d, self.N, self.Y, self.A0, self.inclusions = d, np.full(d, 5), np.ones(d), np.eye(d), []
        self.__dict__.update(kw)


@pytest.mark.parametrize("d", [0, 1])
def test_other_dimensions_reach_the_library(bd, d):
    """The library refuses them by its status; the binding only passes them on."""
    p, keep = bd.problem_struct(Description(d))
    assert p.d == d and list(p.N) == [5] * d + [1] * (3 - d) and list(p.A0) == [1.0 * (d == 1)] + [0.0] * 8


@pytest.mark.parametrize("kw", [dict(d=4), dict(d=2, N=np.full(3, 5)), dict(d=3, Y=np.ones(2)), dict(d=2, A0=np.eye(3)),
                                dict(d=2, inclusions=[ms.Inclusion("box", np.zeros(2), np.ones(4), np.eye(2))]),
                                dict(d=2, inclusions=[ms.Inclusion("box", np.zeros(3), np.ones(2), np.eye(2))]),
                                dict(d=2, bitmap=np.ones(3)), dict(d=2, bitmap=np.ones((3, 4, 5)))],
                         ids=lambda kw: ",".join(kw))
def test_shapes_that_do_not_fit_are_value_errors(bd, kw):
    with pytest.raises(ValueError):
        bd.problem_struct(Description(**kw))


def test_other_number_types(bd):
    """Complex values keep their real part (numpy warns), as every array that is assigned to floats."""
    with pytest.warns(np.exceptions.ComplexWarning):
        p, keep = bd.problem_struct(Description(2, Y=np.array([1 + 1j, 2.0]), A0=np.eye(2) * (3 + 0j)))
    assert list(p.Y) == [1.0, 2.0, 1.0] and list(p.A0)[:5] == [3.0, 0.0, 0.0, 0.0, 3.0]
    p, keep = bd.problem_struct(Description(2, Y=np.array([2.0]), N=np.array([7])))
    assert list(p.Y) == [2.0, 2.0, 1.0] and list(p.N) == [7, 7, 1]
