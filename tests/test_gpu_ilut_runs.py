"""ILUT by the length of its runs (stretches of rows that each couple to the row before): orderings without grid lines,
whose runs are one row, and one chain of millions of rows."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_1606_00541_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(A):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in A]


def reordered(A, order):
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


def coloured(A, m):
    """Eight colours, by the parity of the three coordinates: no row couples to one of its colour."""
    g = np.arange(m ** 3)
    return reordered(A, np.argsort(g % m % 2 + 2 * (g // m % m % 2) + 4 * (g // m ** 2 % 2), kind="stable"))


def test_runs_of_one_row_keep_every_warp():
    """The 27-point 64^3 in eight colours takes about as long as in its natural order (8.3, 9.2 ms); dealt to groups of eight warps, seven
    of which then have no row, 4 times."""
    from paper_1606_00541_gb300 import hec
    A = synth.stencil27_jitter(64, seed=1)
    times = []
    for B in (dev(A), dev(coloured(A, 64))):
        best = float("inf")
        for _ in range(4):
            torch.cuda.synchronize()
            t = time.perf_counter()
            hec.ilut_factor(*B, p=10, tol=1e-3)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        times.append(best)
    assert times[1] <= 2.5 * times[0], times


def test_coloured_factors_bitwise():
    from paper_1606_00541_gb300 import hec
    A = coloured(synth.stencil27_jitter(18, seed=2), 18)
    for got, ref in zip(hec.ilut_factor(*dev(A), p=8, tol=1e-3), oracle.ilut(A, 8, 1e-3)):
        for x, y in zip(got.tensors(), ref):
            assert np.array_equal(x.cpu().numpy(), y)


def test_one_chain_of_millions_of_rows():
    """A band of seven diagonals: with half of the matrix in flight, the last warps wait 11 seconds for the rows before
    theirs.  A wait gives up only when no row has been published for two.  The leading factors against the oracle's."""
    from paper_1606_00541_gb300 import hec
    n, lead = 5_000_000, 5000
    cols = torch.arange(n, device="cuda")[:, None] + torch.arange(-3, 4, device="cuda")
    inside = (cols >= 0) & (cols < n)
    v = -torch.rand(n, 7, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(3))
    v[:, 3] = 6.0
    rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rp[1:] = inside.sum(1).cumsum(0)
    A = rp, cols[inside].to(torch.int32), v[inside]
    L, U = hec.ilut_factor(*A, p=3, tol=0.0)
    first = inside[:lead] & (cols[:lead] < lead)
    B = [np.concatenate([[0], first.sum(1).cumsum(0).cpu().numpy()]).astype(np.int32),
         cols[:lead][first].cpu().numpy().astype(np.int32), v[:lead][first].cpu().numpy()]
    rows = lead - 8  # the last rows of the block lack columns
    for got, ref in zip((L, U), oracle.ilut(B, 3, 0.0)):
        rp, ci, va = got.tensors()
        k = int(ref[0][rows])
        assert np.array_equal(rp[:rows + 1].cpu().numpy(), ref[0][:rows + 1])
        assert np.array_equal(ci[:k].cpu().numpy(), ref[1][:k]) and np.array_equal(va[:k].cpu().numpy(), ref[2][:k])
