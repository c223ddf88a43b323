"""Which plans get the range schedule, and what a plan that is declined it costs."""
import numpy as np
import pytest
import torch

from paper_1606_00541_gb300 import synth
from test_gpu_range import FACTORS, _box

pytestmark = pytest.mark.gpu


def dev(A):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in A]


def packed(hec, T, uplo, w=-1, vdt="f64"):
    lv = hec.sptrsv_analyze(T[0], T[1], uplo)
    return hec.hec_from_csr(*T, levels=lv, ell_width=w, vdt=vdt), lv


def launches(hec, f):
    before = hec.launch_count()
    out = f()
    return hec.launch_count() - before, out


def test_declined_plan_builds_no_tables():
    """Most entries of a random matrix lie in another range: three launches (chunk counts, costs, a pass over the columns) beside
    those of a plan that was given a shape, and no table."""
    from paper_1606_00541_gb300 import hec
    T = hec.ilu_factor(*dev(synth.random_sparse(3000, 0.002, 4)), k=0)[0].tensors()
    H, lv = packed(hec, T, 0)
    base, _ = launches(hec, lambda: hec.sptrsv_plan_create(H, lv, block_threads=256))
    own, plan = launches(hec, lambda: hec.sptrsv_plan_create(H, lv))
    b = torch.ones(3000, dtype=torch.float64, device="cuda")
    assert launches(hec, lambda: hec.sptrsv_lower(plan, b))[0] == 2  # the global schedule: fill and sweep
    assert own - base == 3


PATHS = {  # name: (L and U, slab width)
    **{name: (lambda hec, make=make, k=k: hec.ilu_factor(*dev(make()), k=k), w) for name, (make, k, w) in FACTORS.items()},
    "lines_97": (lambda hec: hec.ilu_factor(*dev(_box(97, 20, 23)), k=0), -1),   # a level's rows 96 apart: padded words
    "lines_32": (lambda hec: hec.ilu_factor(*dev(_box(32, 40, 23)), k=0), -1),   # 31 apart: padding would collide
    "plane_513": (lambda hec: hec.ilu_factor(*dev(synth.poisson2d_5pt(513, 90)), k=0), -1),
    "plane_65": (lambda hec: hec.ilu_factor(*dev(synth.poisson2d_5pt(65, 190)), k=0), -1),
    "27pt_34": (lambda hec: hec.ilu_factor(*dev(synth.stencil27_jitter(34, seed=3)), k=0), -1),  # two lanes a row, 32 apart
    "box_w4": (lambda hec: hec.ilu_factor(*dev(_box(19, 23, 17)), k=0), 4),
    "ilut_w8": (lambda hec: hec.ilut_factor(*dev(_box(19, 23, 17)), p=10, tol=1e-4), 8),  # four partial sums, two slots a wait
}


@pytest.mark.parametrize("vdt", ["f64", "f32"])
@pytest.mark.parametrize("name", list(PATHS))
def test_ranges_asked_for_equal_global_bitwise(name, vdt):
    """Every factor on the range kernels, whether the estimates would choose them or not."""
    from paper_1606_00541_gb300 import hec
    make, w = PATHS[name]
    for uplo, h in enumerate(make(hec)):
        H, lv = packed(hec, h.tensors(), uplo, w, vdt)
        solve = (hec.sptrsv_lower, hec.sptrsv_upper)[uplo]
        n = lv.n
        plans = [hec.sptrsv_plan_create(H, lv, schedule=s) for s in ("range", "global")]
        hec.sptrsv_plan_check(plans[0])
        for seed in range(2):
            b = torch.as_tensor(synth.uniform_vector(n, seed), device="cuda")
            (ran, x), (ran2, y) = (launches(hec, lambda: solve(p, b)) for p in plans)
            assert (ran, ran2) == (1, 2) and torch.equal(x, y)
        assert hec.hec_sync_status(plans[0]) == hec.OK


@pytest.mark.parametrize("case", ["several_ranges", "two_lanes"])
def test_unpublished_row_ends_the_waits(case):
    """A row whose word never comes, in a factor of several ranges and in one with two lanes a row: the sweep ends with a
    timeout, and the next one, of a sound plan, is right."""
    from paper_1606_00541_gb300 import hec
    A = synth.poisson2d_5pt(201, 199) if case == "several_ranges" else synth.stencil27_jitter(21, seed=3)
    T = hec.ilu_factor(*dev(A), k=0)[0].tensors()
    H, lv = packed(hec, T, 0)
    n = lv.n
    b = torch.as_tensor(synth.uniform_vector(n, 3), device="cuda")
    bad = hec.sptrsv_plan_create(H, lv, schedule="range", wait_cycles=5_000_000, debug_unpublished_row=n // 3)
    assert launches(hec, lambda: hec.sptrsv_lower(bad, b))[0] == 1
    assert hec.hec_sync_status(bad) == hec.STATUS_NAMES.index("TIMEOUT")
    good, ref = (hec.sptrsv_plan_create(H, lv, schedule=s) for s in ("range", "global"))
    assert torch.equal(hec.sptrsv_lower(good, b), hec.sptrsv_lower(ref, b))


def test_dense_blocks_take_the_ranges():
    """Blocks of 48 rows, all entries beyond the slab in the row's own range: the long tails are short waits there."""
    from paper_1606_00541_gb300 import hec
    m, b = 500, 48
    n = m * b
    rp = np.arange(n + 1, dtype=np.int32) * b
    ci = (np.arange(n)[:, None] // b * b + np.arange(b)).astype(np.int32).ravel()
    v = synth._rng(1).uniform(-1.0, 1.0, n * b)
    v[ci == np.repeat(np.arange(n), b)] = 1.5 * b
    T = hec.ilu_factor(*dev((rp, ci, v)), k=0)[0].tensors()
    H, lv = packed(hec, T, 0)
    plan, ref = hec.sptrsv_plan_create(H, lv), hec.sptrsv_plan_create(H, lv, schedule="global")
    x = torch.ones(n, dtype=torch.float64, device="cuda")
    (ran, y), (_, z) = (launches(hec, lambda: hec.sptrsv_lower(p, x)) for p in (plan, ref))
    assert ran == 1 and torch.equal(y, z)
