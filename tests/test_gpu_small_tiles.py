"""Products with few tiles take tiles of 64 rows; the three-pass conversion copies pairs of lines where the operand's alignment
allows it.  Both at the sizes, strides and offsets where they change over, bit for bit the oracle's result."""
import numpy as np
import pytest

import synth_inputs as syn
from oracle import oz_oracle as ozo

pytestmark = pytest.mark.gpu

OSET = {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}


@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("S", "int8"), ("E", "fp8"), ("A", "int8"), ("A", "int8n")])
@pytest.mark.parametrize("m,n,k", [(1, 129, 5), (63, 256, 130), (65, 130, 300), (192, 200, 257), (257, 300, 128), (321, 129, 1100), (500, 40, 96)])
def test_few_tiles(set_name, sub, m, n, k):
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + 3 * n + 5 * k)
    A, B = syn._draw(rng, m, k, "lognormal:0.5"), syn._draw(rng, k, n, "normal")
    C0 = np.asfortranarray(rng.standard_normal((m, n)))
    got, st = gh.dgemm(A, B, set_name, gh.route(sub), -1.0, 1.0, C0)
    want = ozo.dgemm(A, B, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS, -1.0, 1.0, C0)
    assert st == 0 and (got == want).all()


@pytest.mark.parametrize("m,n,k", [(16, 16, 128), (33, 17, 129), (15, 40, 7), (50, 260, 384), (201, 99, 250)])
@pytest.mark.parametrize("pad,offset", [(0, 0), (1, 0), (2, 1), (3, 1)])
def test_three_pass_conversion_on_views(m, n, k, pad, offset):
    """The accurate rule takes the scans and the tile conversion at every size.  Operands inside a larger block: leading dimensions
    of either parity, a first element on a 16-byte boundary or not, and NaN around them that must not be read as data."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + n + k + pad)
    A, B = syn._draw(rng, m, k, "normal"), syn._draw(rng, k, n, "normal")
    if m > 15:
        A[3, :] = 0.0
        A[7, k // 2] = np.nan
    rt = gh.route("fp8", rule="ACCURATE")
    want = ozo.dgemm(A, B, ozo.SET_S, ozo.QUANT_RN, ozo.SCALE_ACCURATE)
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, oz.OZ_SET_S, rt))

    def inside(X):
        rows, cols = X.shape
        ld = rows + pad
        flat = torch.full((ld * cols + 2,), float("nan"), dtype=torch.float64, device="cuda")
        flat[offset: offset + ld * cols].view(cols, ld)[:, :rows] = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
        return flat, flat[offset:], ld
    (keepA, dA, lda), (keepB, dB, ldb) = inside(A), inside(B)
    dC = torch.zeros((n, m), dtype=torch.float64, device="cuda")
    oz.check(oz.oz_dgemm_ex(m, n, k, 1.0, dA, lda, dB, ldb, 0.0, dC, m, oz.OZ_SET_S, rt), "oz_dgemm_ex")
    gh.sync_status()
    got = gh.from_dev(dC)
    assert (np.isnan(got) == np.isnan(want)).all()
    assert (got[~np.isnan(want)] == want[~np.isnan(want)]).all()


@pytest.mark.parametrize("k", [1, 128, 129, 384, 385, 896, 1025])
@pytest.mark.parametrize("m,n", [(700, 600), (700, 100), (1100, 1290)])
@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("E", "int8"), ("A", "fp8")])
def test_square_chains(set_name, sub, m, n, k):
    """The two chains of a square modulus over 1, 2, 3, 4, 7 and 9 chunks of k (a pair starts with two chunks and goes on one at a time;
    its ring holds three), several products per pair of blocks, in one block where there are few columns."""
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(k + m + n)
    A, B = syn._draw(rng, m, k, "normal"), syn._draw(rng, k, n, "lognormal:0.5")
    got, st = gh.dgemm(A, B, set_name, gh.route(sub) | oz.OZ_ACC_SEPARATE)
    assert st == 0 and (got == ozo.dgemm(A, B, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS)).all()
