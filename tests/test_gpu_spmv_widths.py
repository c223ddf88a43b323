"""The single-right-hand-side product by slab width: every width with an instance of its own, the first beyond, and the
three scalings, against the oracle's serial product (FP64, sums of at most 24 terms)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu

A = synth.random_sparse(900, 0.015, 9)  # 4 to 24 entries a row


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.5, 0.0), (-1.0, 1.0)])
@pytest.mark.parametrize("w", list(range(0, 19)))
def test_spmv_by_width(w, alpha, beta):
    from paper_1606_00541_gb300 import hec
    H = hec.hec_from_csr(*[torch.as_tensor(a, device="cuda") for a in A], ell_width=w)
    x, y = synth.uniform_vector(900, 1), synth.uniform_vector(900, 2)
    got = hec.spmv(H, torch.as_tensor(x, device="cuda"), torch.as_tensor(y, device="cuda"), alpha=alpha, beta=beta)
    ref = alpha * oracle.spmv(A, x) + beta * y
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-14 * np.max(np.abs(ref))
