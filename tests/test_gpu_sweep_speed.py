"""Sweeps against one another in time, where a wait's polls decide it: a schedule or value type that moves fewer words
must not be the slower one.  The fastest of several passes on each side; margins are far from both figures measured."""
import numpy as np
import pytest
import torch

from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(A):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in A]


def permuted(A, order):
    """The matrix with row and column order[i] in place i."""
    rp, ci, v = A
    n = len(rp) - 1
    new = np.empty(n, np.int64)
    new[order] = np.arange(n)
    r, c = new[np.repeat(np.arange(n), np.diff(rp))], new[ci]
    at = np.lexsort((c, r))
    out = np.zeros(n + 1, np.int32)
    out[1:] = np.cumsum(np.bincount(r, minlength=n))
    return out, c[at].astype(np.int32), v[at]


def fastest(calls, reps=12):
    """Of each call: the least time of `reps` passes, taken in turn."""
    best = [float("inf")] * len(calls)
    for f in calls:
        f()
    for _ in range(reps):
        for i, f in enumerate(calls):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            f()
            b.record()
            b.synchronize()
            best[i] = min(best[i], a.elapsed_time(b) * 1e3)
    return best


def apply_of(hec, L, U, n, nrhs=1, **kw):
    s = hec.IluSolver(L, U, max_nrhs=nrhs, **kw)
    b = torch.ones((n, nrhs) if nrhs > 1 else n, dtype=torch.float64, device="cuda")
    z = torch.empty_like(b)
    return s, lambda: s.apply(b, z)


def test_one_lane_a_row_of_scattered_words():
    """ILUT(10, 1e-3) of the 27-point 64^3, one lane a row: FP32 takes 0.7 times as long as FP64 (1.5 / 2.3 ms); with all the
    warps that fit, each with eight words a lane outstanding, 1.5 times."""
    from paper_1606_00541_gb300 import hec
    n = 64 ** 3
    L, U = [h.tensors() for h in hec.ilut_factor(*dev(synth.stencil27_jitter(64, seed=1)), p=10, tol=1e-3)]
    t64, t32 = fastest([apply_of(hec, L, U, n, vdt=vdt, lanes_per_row=1)[1] for vdt in ("f64", "f32")])
    assert t32 <= 1.1 * t64, (t32, t64)


@pytest.mark.parametrize("lanes", [4, 8])
def test_wide_levels_get_all_warps(lanes):
    """ILU(0) of a random ordering of the 7-point 100^3, levels of thousands of rows, several lanes a row: the plan's own shape
    against 256 threads and as many blocks as fit (16 warps an SM: up to twice as long on such levels)."""
    from paper_1606_00541_gb300 import hec
    n = 100 ** 3
    A = dev(permuted(synth.poisson3d_7pt(100), synth._rng(5).permutation(n)))
    L, U = [h.tensors() for h in hec.ilu_factor(*A, k=0)]
    own, full = fastest([apply_of(hec, L, U, n, vdt="f32", lanes_per_row=lanes, **kw)[1] for kw in ({}, dict(block_threads=256))])
    assert own <= 1.25 * full, (own, full)


def test_partitioned_fp64_of_six_slots():
    """ILU(1) of the 7-point 100^3 in 76 parts.  FP64 takes about 1.9 times as long as FP32 (1790 / 940 us); with its eight
    words polled at once, and spilled, 2.8 times."""
    from paper_1606_00541_gb300 import hec
    n = 100 ** 3
    L, U = [h.tensors() for h in hec.ilu_factor(*dev(synth.poisson3d_7pt(100)), k=1)]
    part = (torch.arange(n, device="cuda") * 76 // n).to(torch.int32)
    calls = []
    for vdt in ("f64", "f32"):
        s, f = apply_of(hec, L, U, n, vdt=vdt)
        s.partition(part, 76, threads=512)
        calls.append(f)
    t64, t32 = fastest(calls)
    assert t64 <= 2.3 * t32, (t64, t32)


def red_black(A, m):
    g = np.arange(m ** 3)
    return permuted(A, np.argsort((g % m + g // m % m + g // m ** 2) % 2, kind="stable"))


@pytest.mark.parametrize("case", ["long_tails", "streams"])
def test_default_schedule_is_not_the_slower_one(case):
    """A default plan against the global schedule (which a plan for two right-hand sides has).  Long tails: ILU(1) of the
    red-black 7-point 100^3, FP32 (range schedule 1200 us, global 860); a factor that does not stay in the caches: ILUT of the
    27-point 100^3, BF16 (2080, 1750)."""
    from paper_1606_00541_gb300 import hec
    n = 100 ** 3
    if case == "long_tails":
        F, vdt = hec.ilu_factor(*dev(red_black(synth.poisson3d_7pt(100), 100)), k=1), "f32"
    else:
        F, vdt = hec.ilut_factor(*dev(synth.stencil27_jitter(100, seed=1)), p=10, tol=1e-3), "bf16"
    L, U = [h.tensors() for h in F]
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    default, two = (hec.IluSolver(L, U, vdt=vdt, max_nrhs=k) for k in (1, 2))
    t1, t2 = fastest([lambda: default.apply(b), lambda: two.apply(b)])
    assert t1 <= 1.1 * t2, (t1, t2)


@pytest.mark.parametrize("nx", [65, 97])
def test_range_words_out_of_one_bank(nx):
    """Lines of 64 k + 1 or 96 + 1 points: the rows of a level lie 64 or 96 words apart in a range's shared solution, one bank without
    padding (97 x 76 x 83, FP64, L+U apply 900 us; the global schedule 520, with padding 290)."""
    from paper_1606_00541_gb300 import hec
    n = nx * 76 * 83
    A = synth.fv7_lognormal_box(nx, 76, 83, np.ones(n))
    L, U = [h.tensors() for h in hec.ilu_factor(*dev(A), k=0)]
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    default, two = (hec.IluSolver(L, U, max_nrhs=k) for k in (1, 2))
    t1, t2 = fastest([lambda: default.apply(b), lambda: two.apply(b)])
    assert t1 <= 0.9 * t2, (t1, t2)
