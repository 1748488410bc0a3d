"""GPU parity of the unvectorised SpMM and SDDMM (any width and alignment): integer inputs, bit for bit.

Loads are 1 to 8 bytes, as the width, the leading dimension and the base address allow; the widths
cross every number of units per lane and of lanes per entry, and the last pass past 256 units.
"""
import numpy as np
import pytest

import gen
import oracle
from _util import dev

pytestmark = pytest.mark.gpu

LENGTHS = np.r_[np.tile([0, 1, 3, 4, 5, 8, 31, 32, 33, 64, 65, 100], 40), [700, 0, 1500]]


@pytest.fixture(scope="module")
def gb():
    import paper_2604_27985_gb300 as g

    return g


def stored(x, dtype, base, ld):
    """x with elements of the dtype, `base` elements past an aligned address, rows ld apart."""
    import torch

    kind = {"f32": torch.float32, "bf16": torch.bfloat16, "e4m3": torch.uint8}[dtype]
    flat = torch.zeros(base + x.shape[0] * ld, dtype=kind, device="cuda")
    v = flat[base:].view(x.shape[0], ld)[:, :x.shape[1]]
    v[:] = dev(oracle.e4m3_round(x)) if dtype == "e4m3" else dev(x).to(kind)
    return v


@pytest.mark.parametrize("dtype", ["f32", "bf16", "e4m3"])
@pytest.mark.parametrize("N,base,pad", [(1, 0, 0), (7, 0, 0), (31, 0, 0), (33, 1, 0), (50, 0, 2), (65, 0, 0), (100, 1, 0),
                                        (102, 2, 0), (129, 0, 3), (200, 0, 1), (255, 0, 0), (260, 4, 2), (515, 0, 0)])
def test_units_integers_bit_exact(gb, dtype, N, base, pad):
    import torch

    A = gen.csr_from_lengths(LENGTHS, 1600, seed=800)
    M, K = A.M, A.K
    vals = gen.vals_int(A.nnz, 801, -4, 4)
    B, X = gen.dense_int(K, N, 802, -4, 4), gen.dense_int(M, N, 803, -4, 4)
    one = lambda n: torch.ones(n, device="cuda") if dtype == "e4m3" else None
    rp, ci = dev(A.rowptr), dev(A.colidx)
    a = dev(oracle.e4m3_round(vals)) if dtype == "e4m3" else dev(vals).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    b, x = stored(B, dtype, base, N + pad), stored(X, dtype, base, N + pad)
    C = gb.spmm(rp, ci, a, b, a_scale=one(M), b_scale=one(K), variant="scalar")
    assert np.array_equal(C.cpu().numpy().astype(np.float64), oracle.spmm(A.rowptr, A.colidx, vals, B)[0])
    out = gb.sddmm(rp, ci, dev(vals), x, b, x_scale=one(M), y_scale=one(K), variant="scalar")
    assert np.array_equal(out.cpu().numpy().astype(np.float64), oracle.sddmm(A.rowptr, A.colidx, vals, X, B)[0])


def test_units_leave_infinities_where_they_are(gb):
    """Lanes past a row's width read its first element and must not let it into a sum."""
    A = gen.csr_from_lengths(LENGTHS, 1600, seed=810)
    vals = gen.vals_int(A.nnz, 811)
    B, X = gen.dense_int(1600, 77, 812), gen.dense_int(A.M, 77, 813)
    want = oracle.spmm(A.rowptr, A.colidx, vals, B)[0]
    B[5, 0] = np.inf
    C = gb.spmm(dev(A.rowptr), dev(A.colidx), dev(vals), dev(B), variant="scalar").cpu().numpy()
    assert np.array_equal(C[:, 1:].astype(np.float64), want[:, 1:])
    out = gb.sddmm(dev(A.rowptr), dev(A.colidx), dev(vals), dev(X), dev(B), variant="scalar").cpu().numpy()
    clean = A.colidx != 5
    B[5, 0] = 0
    assert np.array_equal(out[clean].astype(np.float64), oracle.sddmm(A.rowptr, A.colidx, vals, X, B)[0][clean])


@pytest.mark.parametrize("dtype", ["f32", "bf16", "e4m3"])
@pytest.mark.parametrize("N,base", [(24, 0), (66, 1), (96, 1), (97, 0), (120, 0), (127, 0), (128, 1), (161, 0), (192, 1), (193, 0), (257, 0)])
def test_spmm_elements_bit_exact(gb, dtype, N, base):
    """Single elements: three and four columns a lane, one and four entries in flight, whole and cut passes; units
    halved so that half of the lanes have one (N = 24, 120)."""
    import torch

    A = gen.csr_from_lengths(LENGTHS, 1600, seed=815)
    vals, B = gen.vals_int(A.nnz, 816, -4, 4), gen.dense_int(1600, N, 817, -4, 4)
    one = lambda n: torch.ones(n, device="cuda") if dtype == "e4m3" else None
    a = dev(oracle.e4m3_round(vals)) if dtype == "e4m3" else dev(vals).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    C = gb.spmm(dev(A.rowptr), dev(A.colidx), a, stored(B, dtype, base, N), a_scale=one(A.M), b_scale=one(1600),
                variant="scalar")
    assert np.array_equal(C.cpu().numpy().astype(np.float64), oracle.spmm(A.rowptr, A.colidx, vals, B)[0])


@pytest.mark.parametrize("dtype,Kd", [("f32", 17), ("f32", 22), ("bf16", 33), ("e4m3", 36), ("e4m3", 72), ("e4m3", 104)])
def test_sddmm_short_rows_bit_exact(gb, dtype, Kd):
    """Rows of one to five entries on either side of the line between one lane per entry and the units."""
    import torch

    for mean in (2, 5):
        A = gen.csr_from_lengths(np.tile(np.arange(2 * mean + 1), 300), 900, seed=820)
        vals = gen.vals_int(A.nnz, 821, -4, 4)
        X, Y = gen.dense_int(A.M, Kd, 822, -4, 4), gen.dense_int(A.K, Kd, 823, -4, 4)
        one = lambda n: torch.ones(n, device="cuda") if dtype == "e4m3" else None
        out = gb.sddmm(dev(A.rowptr), dev(A.colidx), dev(vals), stored(X, dtype, 0, Kd), stored(Y, dtype, 0, Kd),
                       x_scale=one(A.M), y_scale=one(A.K), variant="scalar")
        assert np.array_equal(out.cpu().numpy().astype(np.float64), oracle.sddmm(A.rowptr, A.colidx, vals, X, Y)[0])
