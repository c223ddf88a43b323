"""The sweeps by slab width (three, four and more slots in registers, further slots, tails) in the global and the
partitioned kernels, one and several right-hand sides, with infinities and NaN in the right-hand side reaching exactly
the rows that depend on them."""
import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu

BOX = synth.fv7_lognormal_box(13, 17, 11, synth._rng(1).uniform(0.5, 2.0, 13 * 17 * 11))
N = 13 * 17 * 11
LO, UP = oracle.iluk(BOX, 1)  # up to six entries beside the diagonal


def _plan(hec, w, vdt, nrhs, parts, uplo):
    T = [torch.as_tensor(a, device="cuda") for a in (LO, UP)[uplo]]
    lv = hec.sptrsv_analyze(T[0], T[1], uplo)
    p = hec.sptrsv_plan_create(hec.hec_from_csr(*T, levels=lv, ell_width=w, vdt=vdt), lv, nrhs, block_threads=128,
                               lanes_per_row=1)
    if parts:
        hec.sptrsv_plan_partition(p, None, parts, 128)
    return p


@pytest.mark.parametrize("uplo", [0, 1])
@pytest.mark.parametrize("nrhs,parts", [(1, 0), (1, 1), (1, 7), (3, 0), (16, 0)])
@pytest.mark.parametrize("w", [0, 2, 3, 4, 6, 9])
def test_slab_widths(w, nrhs, parts, uplo):
    from paper_1606_00541_gb300 import hec
    p = _plan(hec, w, "f64", nrhs, parts, uplo)
    b = synth.uniform_vector(N, 3, nrhs=nrhs)
    x = (hec.sptrsv_lower, hec.sptrsv_upper)[uplo](p, torch.as_tensor(b, device="cuda")).cpu().numpy().reshape(N, -1)
    for q in range(nrhs):
        ref = (oracle.lower_solve, oracle.upper_solve)[uplo]((LO, UP)[uplo], b.reshape(N, -1)[:, q])
        assert np.max(np.abs(x[:, q] - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("vdt", ["f64", "f32"])
@pytest.mark.parametrize("w,parts", [(3, 5), (4, 5), (6, 5), (3, 0), (6, 0)])
def test_nonfinite_values_stay_in_their_rows(w, parts, vdt, value):
    """A slot that a row does not use (its padding, a dependency in another part) must not carry a value in."""
    from paper_1606_00541_gb300 import hec
    p = _plan(hec, w, vdt, 1, parts, 0)
    b = synth.uniform_vector(N, 5)
    b[1000] = value
    x = hec.sptrsv_lower(p, torch.as_tensor(b, device="cuda")).cpu().numpy()
    rp, ci, _ = LO
    reached = np.zeros(N, bool)
    for i in range(N):
        reached[i] = i == 1000 or reached[ci[rp[i]:rp[i + 1] - 1]].any()
    assert np.array_equal(~np.isfinite(x), reached)
