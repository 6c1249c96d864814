"""The FP64 near fields' log, reciprocal and reciprocal square root (fp64_math.cuh), one value at a time.

One unit charge at the origin and zero charges at (x, 0) in a tree of one cell: the potential (or the field) at x
is the function of the one distance alone, as every other pair adds a zero.  Distances: all exponents, 1 +- 2^-k,
both ends and the centre of every interval of the logarithm's table, random ones about 1, and r^2 at the ends of
the normal range and below it.  The reference is the function of fl(x^2) in extended precision.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def distances(case):
    rng = np.random.default_rng(8700)
    k = np.arange(1, 53)
    if case == "about 1":
        x = np.concatenate(([1.0], 1.0 + 2.0 ** -k, 1.0 - 2.0 ** -k, 1.0 + (rng.random(1500) - 0.5) * 2.0 ** -rng.integers(0, 40, 1500)))
    elif case == "table":   # r^2 at multiples of 2^-10 within [1/2, 2], two units either side
        edge = np.sqrt(np.arange(512, 2049) / 1024.0)
        x = np.concatenate((edge, edge * (1.0 + 2.0 ** -51), edge * (1.0 - 2.0 ** -51)))
    elif case == "exponents":
        x = (1.0 + rng.random(3000)) * 2.0 ** rng.integers(-510, 511, 3000)
    else:   # r^2 below 2^-1022, at the first normal numbers, and at the last ones
        x = np.concatenate((2.0 ** np.arange(-530.0, -505.0), 1.3 * 2.0 ** np.arange(-530.0, -505.0), 2.0 ** np.arange(505.0, 512.0),
                            1.3 * 2.0 ** np.arange(505.0, 512.0)))
    return np.unique(x)


CASES = ["about 1", "table", "exponents", "ends"]
BOX = 2.0 ** 513


def system(case, dim):
    x = distances(case)
    pos = np.zeros((x.size + 1, dim))
    pos[1:, 0] = x
    q = np.zeros(x.size + 1)
    q[0] = 1.0
    return x, (x * x).astype(np.longdouble), pos, q


def check(got, ref, units, what):
    ref = np.asarray(ref)
    off = np.abs(got.astype(np.longdouble) - ref) / np.spacing(np.abs(ref).astype(np.float64))
    off = np.where(got == ref, 0.0, off.astype(np.float64))
    assert np.all(off <= units), f"{what}: {off.max():.3g} units, entry {np.argmax(off)}"


@pytest.mark.parametrize("case", CASES)
def test_log(case):
    """A table entry (one unit of a value at most twice the result) and three roundings: within 4 units."""
    from gpu_util import to_dev
    from paper_2009_00767_gb300 import binding
    x, r2, pos, q = system(case, 2)
    txy, tq = to_dev(pos, q)
    with binding.Plan(q.size, 0, 4, BOX, "fp64") as plan:
        phi = plan.potential(txy, tq).cpu().numpy()[1:]
    check(phi, 0.5 * np.log(r2), 4, f"log, {case}")


@pytest.mark.parametrize("case", CASES)
def test_reciprocal(case):
    """x fl(1 / r^2): 1 / r^2 within one unit and the product's rounding, so within 2 units of a value up to twice
    the spacing: 4.  A subnormal 1 / r^2 has no more than its own spacing."""
    from gpu_util import to_dev
    from paper_2009_00767_gb300 import binding
    x, r2, pos, q = system(case, 2)
    # 1 / r^2 overflows below 2^-1022; zero charges that are as close to each other would add 0 times infinity, so
    # the smallest distances come one to a call
    keep = r2 >= np.longdouble(2.0) ** -1022
    together = np.concatenate(([True], x >= 2.0 ** -450))
    e = np.zeros(x.size)
    with binding.Plan(int(together.sum()), 0, 4, BOX, "fp64") as plan:
        _, field = plan.potential_field(*to_dev(pos[together], q[together]))
    e[together[1:]] = -field.cpu().numpy()[1:, 0]
    with binding.Plan(2, 0, 4, BOX, "fp64") as plan:
        for i in np.flatnonzero(keep & ~together[1:]):
            _, field = plan.potential_field(*to_dev(pos[[0, i + 1]], q[[0, i + 1]]))
            e[i] = -field.cpu().numpy()[1, 0]
    ref = x.astype(np.longdouble) / r2
    slack = np.where(r2 > np.longdouble(2.0) ** 1022, x.astype(np.longdouble) * np.longdouble(2.0) ** -1074, 0.0)
    near = np.clip(e.astype(np.longdouble), ref - slack, ref + slack)   # the nearest value that is allowed exactly
    check(e[keep], near[keep], 4, f"reciprocal, {case}")


@pytest.mark.parametrize("case", CASES)
def test_reciprocal_square_root(case):
    """x y0, e and the last FMA round, and the series' remainder is below them: within 4 units."""
    from gpu_util import to_dev
    from paper_2009_00767_gb300 import binding
    x, r2, pos, q = system(case, 3)
    keep = r2 > 0
    tpos, tq = to_dev(pos, q)
    with binding.LagPlan(3, q.size, 0, BOX, "node_f64") as plan:
        phi = plan.potential(tpos, tq).cpu().numpy()[1:]
    check(phi[keep], 1.0 / np.sqrt(r2[keep]), 4, f"reciprocal square root, {case}")
