"""The factorization kernels at the shapes that decide their work split: ILU(0) rows at and beyond the limits of
the thread-per-row elimination, with pivots that change other pivots' entries, at sizes around a warp and beyond
the resident threads; ILUT on runs of one row, of a grid line and longer than a run's limit."""
import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(A):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in A]


def host(h):
    return [t.cpu().numpy() for t in h.tensors()]


def _banded(n, offsets, seed=0, zero_row=None):
    """Entries at the given column offsets, values U[-1, 1], diagonally dominant."""
    rng = synth._rng(seed)
    rows = [[i + o for o in offsets if 0 <= i + o < n] for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    ci = np.concatenate(rows).astype(np.int32)
    v = rng.uniform(-1.0, 1.0, len(ci))
    row = np.repeat(np.arange(n), np.diff(rp))
    v[ci == row] = 1.5 * len(offsets)
    if zero_row is not None:
        v[row == zero_row] = 0.0
    return rp, ci, v


def _box(nx, ny, nz):
    return synth.fv7_lognormal_box(nx, ny, nz, synth._rng(1).uniform(0.5, 2.0, nx * ny * nz))


ILU0 = {
    "diagonal": lambda: _banded(33, [0]),
    "one_row": lambda: _banded(1, [0]),
    "penta_257": lambda: _banded(257, range(-2, 3)),           # a pivot changes the next pivot's entry
    "hepta_31": lambda: _banded(31, range(-3, 4)),
    "8_entries_4_pivots": lambda: _banded(1000, range(-4, 4)),  # the limits of the thread-per-row kernel
    "9_entries": lambda: _banded(1000, range(-4, 5)),           # beyond them: warp per row
    "8_entries_5_pivots": lambda: _banded(1000, range(-5, 3)),
    "far_offsets": lambda: _banded(3000, [-700, -31, -1, 0, 1, 31, 700]),
    "lines_33": lambda: _box(33, 9, 5),
    "resident": lambda: _box(61, 59, 57),                       # 205,143 rows: more than the resident threads
}


@pytest.mark.parametrize("case", list(ILU0))
def test_ilu0_by_row_shape(case):
    from paper_1606_00541_gb300 import hec
    A = ILU0[case]()
    for got, ref in zip(hec.ilu_factor(*dev(A), k=0), oracle.ilu0(A)):
        rp, ci, v = host(got)
        assert np.array_equal(rp, ref[0]) and np.array_equal(ci, ref[1])
        assert np.max(np.abs(v - ref[2])) <= 1e-12 * np.max(np.abs(ref[2]))


@pytest.mark.parametrize("offsets", [range(-2, 3), range(-4, 5)], ids=["thread_per_row", "warp_per_row"])
def test_ilu0_zero_pivot(offsets):
    from paper_1606_00541_gb300 import hec
    with pytest.raises(hec.HecError) as e:
        hec.ilu_factor(*dev(_banded(500, offsets, zero_row=0)), k=0)
    assert hec.STATUS_NAMES[e.value.status] == "ZERO_PIVOT"


ILUT = {
    "runs_of_one": lambda: _banded(3000, [-64, -2, 0, 2, 64]),   # no row has an entry in the column before its own
    "one_long_run": lambda: _banded(9000, [-1, 0, 1]),           # longer than a run's limit
    "lines_31": lambda: _box(31, 12, 9),
    "few_runs": lambda: _banded(100, [-1, 0, 1]),
    "resident": lambda: synth.stencil27_jitter(34, seed=5),      # 39,304 rows: more than the resident warps
}


@pytest.mark.parametrize("scale", [1e-307, 1e-160, 1e-20, 1e150, 1e300])
@pytest.mark.parametrize("p", [2, 40])
def test_ilut_over_the_exponent_range_bitwise(p, scale):
    """Quotients of the elimination: rows scaled over the range of FP64 (every third row by `scale`), so that some
    pivots, values and quotients leave the range of the corrected reciprocal."""
    A = synth.random_sparse(400, 0.02, 11)
    row = np.repeat(np.arange(400), np.diff(A[0]))
    A = (A[0], A[1], np.where(row % 3 == 0, A[2] * scale, A[2]))
    from paper_1606_00541_gb300 import hec
    for got, ref in zip(hec.ilut_factor(*dev(A), p=p, tol=1e-4), oracle.ilut(A, p, 1e-4)):
        for x, y in zip(host(got), ref):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("case", list(ILUT))
def test_ilut_by_run_shape_bitwise(case):
    from paper_1606_00541_gb300 import hec
    A = ILUT[case]()
    for got, ref in zip(hec.ilut_factor(*dev(A), p=6, tol=1e-3), oracle.ilut(A, 6, 1e-3)):
        for x, y in zip(host(got), ref):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("scale", [1e-300, 1e-20, 1e150])
def test_ilu0_over_the_exponent_range(scale):
    """Warp-per-row elimination of rows scaled over the range of FP64 (every third row by `scale`): the quotients are
    those of the division, so the factors stay within the rounding of a fused update."""
    from paper_1606_00541_gb300 import hec
    A = _banded(600, range(-6, 7))
    row = np.repeat(np.arange(600), np.diff(A[0]))
    A = (A[0], A[1], np.where(row % 3 == 0, A[2] * scale, A[2]))
    for got, ref in zip(hec.ilu_factor(*dev(A), k=0), oracle.ilu0(A)):
        rp, ci, v = host(got)
        assert np.array_equal(rp, ref[0]) and np.array_equal(ci, ref[1]) and np.isfinite(v).all()
        r = np.repeat(np.arange(600), np.diff(rp))
        big = np.maximum.reduceat(np.abs(ref[2]), rp[:-1])[r]  # row by row: the rows differ in scale
        assert np.all(np.abs(v - ref[2]) <= 1e-12 * big)
