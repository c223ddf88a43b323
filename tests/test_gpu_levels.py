"""Level analysis on the patterns that decide how a chunk of 32 rows publishes its levels: grid lines of
fewer, as many and more rows than a chunk, rows with more outside dependencies than one batch, dependencies
inside a chunk that skip the preceding row, and more rows than are in flight at once.  Bit-exact against the
oracle's serial levels and maps."""
import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu


def _lower_upper(A, uplo):
    rp, ci, v = A
    row = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    keep = ci <= row if uplo == 0 else ci >= row
    out = np.zeros_like(rp)
    np.add.at(out, row[keep] + 1, 1)
    return np.cumsum(out).astype(np.int32), ci[keep], v[keep]


def test_width_rule_with_a_long_row():
    """A row of more entries than the row-count histogram's bins: counted again with every bin."""
    from paper_1606_00541_gb300 import hec
    n = 1400
    rp = np.concatenate([np.arange(n), [2 * n - 1]]).astype(np.int32)  # the diagonal, and a full last row
    ci = np.concatenate([np.arange(n - 1), np.arange(n)]).astype(np.int32)
    T = (rp, ci, np.linspace(1.0, 2.0, len(ci)))
    Td = [torch.as_tensor(a, device="cuda") for a in T]
    lv = hec.sptrsv_analyze(Td[0], Td[1], 0)
    ref = oracle.analyze(T, 0)
    H = hec.hec_from_csr(*Td, levels=lv).arrays()
    R = oracle.hec_pack(T, 1, 0, ref["perm"], ref["iperm"])
    assert H["w"] == R["w"]
    for key in ["ell_col", "tptr", "tcol"]:
        assert np.array_equal(H[key].cpu().numpy(), R[key]), key


def _box(nx, ny, nz):
    return synth.fv7_lognormal_box(nx, ny, nz, synth._rng(1).uniform(0.5, 2.0, nx * ny * nz))


CASES = {
    "line31": lambda: _box(31, 9, 5),
    "line32": lambda: _box(32, 9, 5),
    "line33": lambda: _box(33, 9, 5),
    "line5": lambda: _box(5, 7, 11),                      # several lines in one chunk
    "line200": lambda: _box(200, 3, 3),
    "27pt": lambda: synth.stencil27_jitter(9, seed=3),    # 13 dependencies a row
    "27pt_long": lambda: synth.stencil27_jitter(40, seed=3),
    "gaps": lambda: synth.random_sparse(900, 0.02, 7),    # chunks with arbitrary inside dependencies
    "chain": lambda: synth.poisson2d_5pt(3000, 1),        # 3,000 levels: more than one pass of the level sort
    "in_flight": lambda: _box(97, 91, 89),                # 785,603 rows: more than the resident lanes
}


@pytest.mark.parametrize("uplo", [0, 1])
@pytest.mark.parametrize("case", list(CASES))
def test_levels_by_chunk_shape(case, uplo):
    from paper_1606_00541_gb300 import hec
    T = _lower_upper(CASES[case](), uplo)
    lv = hec.sptrsv_analyze(*(torch.as_tensor(a, device="cuda") for a in T[:2]), uplo)
    ref = oracle.analyze(T, uplo)
    assert lv.nlev == ref["nlev"]
    for got, key in zip(lv.arrays(), ["level", "perm", "iperm", "level_ptr"]):
        assert np.array_equal(got.cpu().numpy(), ref[key]), key
