"""The default (range) schedule of single-right-hand-side sweeps against the global one on the same factor: the
same bits for every value type, direction and slab shape, from one row to more rows than one SM's shared memory, on
repeated calls, inside a captured graph and with a preconditioner's gathers and scatters."""
import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(A):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in A]


def _box(nx, ny, nz):
    return synth.fv7_lognormal_box(nx, ny, nz, synth._rng(1).uniform(0.5, 2.0, nx * ny * nz))


FACTORS = {  # name: (matrix, fill level, slab width)
    "one_row": (lambda: synth.poisson2d_5pt(1, 1), 0, -1),
    "31x1": (lambda: synth.poisson2d_5pt(31, 1), 0, -1),
    "chain": (lambda: synth.poisson2d_5pt(5000, 1), 0, -1),        # one row a level
    "2d_64": (lambda: synth.poisson2d_5pt(64), 0, -1),             # one range
    "2d_201x199": (lambda: synth.poisson2d_5pt(201, 199), 0, -1),  # several
    "box": (lambda: _box(40, 33, 27), 0, -1),
    "box_tail": (lambda: _box(19, 23, 17), 0, 1),                  # so long a tail that the default is two lanes a row
    "slim_tail": (lambda: _box(3, 3, 300), 0, 2),                  # a tail entry in some rows
    "box_wide": (lambda: _box(19, 23, 17), 1, 6),                  # eight slots a wait
    "box_fill2": (lambda: _box(19, 23, 17), 2, -1),                # long rows: four partial sums, two lanes a row
    "27pt": (lambda: synth.stencil27_jitter(21, seed=3), 0, -1),   # eight partial sums
    "27pt_one_range": (lambda: synth.stencil27_jitter(9, seed=3), 0, 13),
    "27pt_tail": (lambda: synth.stencil27_jitter(21, seed=3), 0, 6),   # two partial sums and a long tail
    "27pt_w17": (lambda: synth.stencil27_jitter(12, seed=3), 1, 17),   # two waits a row, and a tail
    "box_pad": (lambda: _box(19, 23, 17), 0, 9),                   # slots that every row leaves empty
    "random": (lambda: synth.random_sparse(3000, 0.002, 4), 0, -1),
    "large": (lambda: _box(101, 97, 83), 0, -1),                   # 813,151 rows
}


def _solvers(hec, T, uplo, w, vdt):
    lv = hec.sptrsv_analyze(T[0], T[1], uplo)
    H = hec.hec_from_csr(*T, levels=lv, ell_width=w, vdt=vdt)
    solve = hec.sptrsv_lower if uplo == 0 else hec.sptrsv_upper
    default = hec.sptrsv_plan_create(H, lv)
    shaped = hec.sptrsv_plan_create(H, lv, block_threads=256)  # a caller's shape: the global kernel, same lanes a row
    return default, shaped, solve


@pytest.mark.parametrize("vdt", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name", list(FACTORS))
def test_range_equals_global_bitwise(name, vdt):
    from paper_1606_00541_gb300 import hec
    make, k, w = FACTORS[name]
    A = make()
    n = len(A[0]) - 1
    factors = [h.tensors() for h in hec.ilu_factor(*dev(A), k=k)]
    for uplo, T in enumerate(factors):
        default, shaped, solve = _solvers(hec, T, uplo, w, vdt)
        hec.sptrsv_plan_check(default)
        for seed in range(3):  # the two word buffers in turn
            b = torch.as_tensor(synth.uniform_vector(n, seed), device="cuda")
            assert torch.equal(solve(default, b), solve(shaped, b))
        assert hec.hec_sync_status(default) == hec.OK


def test_range_is_the_default_and_needs_one_launch():
    from paper_1606_00541_gb300 import hec
    T = hec.ilu_factor(*dev(_box(20, 20, 20)), k=0)[0].tensors()
    default, shaped, solve = _solvers(hec, T, 0, -1, "f64")
    b = torch.ones(8000, dtype=torch.float64, device="cuda")
    launches = []
    for plan in (default, shaped):
        before = hec.launch_count()
        solve(plan, b)
        launches.append(hec.launch_count() - before)
    assert launches == [1, 2]  # the global kernel has a fill before it


def test_short_wait_budget_keeps_the_global_schedule():
    """58 levels are estimated at 26 us, 219,240 cycles with the factor of four: a smaller budget, and the plan sweeps
    with the global kernel (two launches), whose waits are shorter."""
    from paper_1606_00541_gb300 import hec
    T = hec.ilu_factor(*dev(_box(20, 20, 20)), k=0)[0].tensors()
    lv = hec.sptrsv_analyze(T[0], T[1], 0)
    H = hec.hec_from_csr(*T, levels=lv)
    b = torch.ones(8000, dtype=torch.float64, device="cuda")
    launches = []
    for budget in (0, 300_000, 200_000):
        plan = hec.sptrsv_plan_create(H, lv, wait_cycles=budget)
        before = hec.launch_count()
        hec.sptrsv_lower(plan, b)
        launches.append(hec.launch_count() - before)
    assert launches == [1, 1, 2]


def test_range_in_a_captured_graph():
    """Replays poll the word buffer the replay before them reset: an odd number of sweeps a graph."""
    from paper_1606_00541_gb300 import hec
    A = _box(23, 21, 19)
    n = len(A[0]) - 1
    L, U = [h.tensors() for h in hec.ilu_factor(*dev(A), k=0)]
    s = hec.IluSolver(L, U)
    b, x = (torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2))
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        hec.sptrsv_lower(s.pL, b, x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hec.sptrsv_lower(s.pL, b, x)
    Lo = [t.cpu().numpy() for t in L]
    for seed in range(4):
        v = synth.uniform_vector(n, seed)
        b.copy_(torch.as_tensor(v))
        graph.replay()
        torch.cuda.synchronize()
        ref = oracle.lower_solve(Lo, v)
        assert np.max(np.abs(x.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("vdt", ["f64", "f32"])
def test_range_in_schwarz_apply(vdt):
    """Gather through ext2glob, y between the factors, restricted scatter."""
    from paper_1606_00541_gb300 import hec
    A = synth.fv7_lognormal(24, seed=2)
    part, ns = synth.grid_boxes(24, (2, 3, 2))
    Ad, pd = dev(A), torch.as_tensor(part, device="cuda")
    r = torch.as_tensor(synth.uniform_vector(24 ** 3, 1), device="cuda")
    z = [hec.RasSolver(Ad, pd, ns, vdt=vdt, **kw).apply(r) for kw in ({}, dict(block_threads=256))]
    assert torch.equal(*z)
