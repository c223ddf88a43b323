"""Which plans get the range schedule, and what a plan that is declined it costs."""
import numpy as np
import pytest
import torch

from paper_1606_00541_gb300 import synth

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
