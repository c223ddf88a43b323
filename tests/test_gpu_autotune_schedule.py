"""What the autotuner reports is what runs, and a plan made from its report runs the same."""
import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(A):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in A]


def sweep_launches(hec, plan, b):
    before = hec.launch_count()
    x = hec.sptrsv_lower(plan, b)
    return hec.launch_count() - before, x


@pytest.mark.parametrize("case,schedule", [("ranges", "range"), ("shaped", "global"), ("long_rows", None), ("parts", "part")])
def test_report_reproduces_the_choice(case, schedule):
    """One launch a sweep for ranges and parts, two (fill and sweep) for the global kernels."""
    from paper_1606_00541_gb300 import hec
    L = oracle.ilu0(synth.stencil27_jitter(16, seed=1) if case == "long_rows" else synth.poisson2d_5pt(64))[0]
    T, n = dev(L), len(L[0]) - 1
    lv = hec.sptrsv_analyze(T[0], T[1], 0)
    H = hec.hec_from_csr(*T, levels=lv)
    plan = hec.sptrsv_plan_create(H, lv, **(dict(schedule="global") if case in ("shaped", "parts") else {}))
    if case == "parts":
        hec.sptrsv_plan_partition(plan, None, 1, 512)
    choice = hec.sptrsv_autotune(plan, 1)
    schedule = schedule or choice["schedule"]  # either may win on long rows
    assert choice["schedule"] == schedule and choice["partitioned"] == (schedule == "part")
    b = torch.as_tensor(synth.uniform_vector(n, 2), device="cuda")
    ran, x = sweep_launches(hec, plan, b)
    assert ran == (2 if schedule == "global" else 1)
    again = hec.sptrsv_plan_create(H, lv, **choice)
    if case == "parts":
        hec.sptrsv_plan_partition(again, None, 1, 512)
    ran2, y = sweep_launches(hec, again, b)
    assert ran2 == ran and torch.equal(x, y)
    ref = oracle.lower_solve(L, b.cpu().numpy())
    assert np.max(np.abs(x.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))


def test_own_shape_is_among_the_candidates():
    """Eight lanes a row on narrow levels: 64 threads, 8 blocks an SM by default (1838 us an L+U apply; the fastest of the other
    shapes 1866), which a tuned plan may not lose."""
    from paper_1606_00541_gb300 import hec
    A = dev(synth.stencil27_jitter(100, seed=1))
    T = hec.ilu_factor(*A, k=0)[0].tensors()
    lv = hec.sptrsv_analyze(T[0], T[1], 0)
    H = hec.hec_from_csr(*T, levels=lv)
    b = torch.ones(100 ** 3, dtype=torch.float64, device="cuda")
    best = {}
    for name in ("own", "tuned"):
        plan = hec.sptrsv_plan_create(H, lv, schedule="global")
        if name == "tuned":
            hec.sptrsv_autotune(plan, 1)
        x = hec.sptrsv_lower(plan, b)
        times = []
        for _ in range(30):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            hec.sptrsv_lower(plan, b, x)
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        best[name] = min(times)
    assert best["tuned"] <= 1.01 * best["own"], best


def test_unknown_schedule_is_refused():
    from paper_1606_00541_gb300 import hec
    T = dev(oracle.ilu0(synth.poisson2d_5pt(8))[0])
    lv = hec.sptrsv_analyze(T[0], T[1], 0)
    H = hec.hec_from_csr(*T, levels=lv)
    import ctypes
    for value in (-1, 4):
        t, out = hec.HecTune(schedule=value), ctypes.c_void_p()
        assert hec._sptrsv_plan_create(H.h, lv.h, 1, ctypes.byref(t), ctypes.byref(out)) == hec.STATUS_NAMES.index("INVALID_ARG")
