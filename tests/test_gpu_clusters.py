"""Deconstruction by clusters: operands above 4 M elements whose lines spread over the shared memory of one to five blocks.  Every
layout that takes the form on either side, lines whose special elements lie in one block's share only, a last strip of a few
lines, odd strides and 8-byte-aligned operands, bit for bit the oracle's result.  The launch counts say that it was this form."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oz_oracle as ozo

pytestmark = pytest.mark.gpu

OSET = {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}
ROUTES = [("S", "fp8"), ("S", "int8"), ("E", "fp8"), ("E", "int8"), ("A", "fp8"), ("A", "int8"), ("A", "int8n")]


def _lines(rng, lines, k, spread=0.0, spikes=True):
    """lines x k with every kind of line that the form treats apart, at both ends of the operand.  spread: the largest exponent
    spread of a line; spikes: with lines of one large element."""
    X = rng.standard_normal((lines, k))
    if spread:
        X *= np.exp(spread * rng.random((lines, 1)) * rng.standard_normal((lines, k)))
    for at in (0, lines - 9):
        X[at] = 0.0
        X[at + 1] *= 2.0 ** -1050                        # subnormals only
        X[at + 2, 3] = np.nan                            # in the first block's share
        X[at + 3, k - 1] = -np.inf                       # in the last one's
        X[at + 4] *= 2.0 ** 950
        X[at + 5] *= 1e-300
        if spikes:
            X[at + 6] = 0.0
            X[at + 6, k - 2] = 5e-324                    # the smallest number, alone
            X[at + 7] *= 2.0 ** -1060
            X[at + 7, k // 2] = 2.0 ** -1030             # the largest subnormal exponent in one share
            X[at + 8] *= 2.0 ** -1040
            X[at + 8, 1] = 1.5                           # one normal number among subnormals
    return X


def _device(X, pad, offset):
    """Column-major copy with `pad` spare rows (NaN) a column, the first element `offset` doubles into the block."""
    import torch
    rows, cols = X.shape
    ld = rows + pad
    flat = torch.full((ld * cols + 2,), float("nan"), dtype=torch.float64, device="cuda")
    flat[offset: offset + ld * cols].view(cols, ld)[:, :rows] = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    return flat[offset:], ld


def _same(got, want):
    assert (np.isnan(got) == np.isnan(want)).all()
    assert (got[~np.isnan(want)] == want[~np.isnan(want)]).all()


@pytest.mark.parametrize("set_name,sub", ROUTES)
@pytest.mark.parametrize("lines,k,pad,offset", [
    (9470, 597, 0, 0),          # one block
    (4699, 1191, 0, 0),         # two, odd leading dimensions on both sides
    (4700, 1190, 0, 1),         # two, off the 16-byte boundary
    (2970, 1893, 2, 0),         # three
    (2266, 2442, 0, 0),         # four
    (1785, 3150, 3, 0),         # five
])
@pytest.mark.parametrize("side", [0, 1])
def test_kept_operand(side, lines, k, pad, offset, set_name, sub):
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(lines + k + side)
    few = 30
    big, small = _lines(rng, lines, k), rng.standard_normal((few, k))
    A, B = (big, small) if side == 0 else (small, big)
    A, B = np.asfortranarray(A), np.asfortranarray(B.T)
    m, n, sid = A.shape[0], B.shape[1], gh.SETS[set_name]
    (dA, lda), (dB, ldb) = _device(A, pad, offset), _device(B, pad, offset)
    gh.ensure_workspace(oz.oz_product_workspace_bytes(m, n, sid))
    for rule, quant in (("CS", "RN"), ("MAXEXP", "TZ")):
        rt = gh.route(sub, quant, rule)
        ops, launches = [], []
        for s, ln, dX, ld in ((0, m, dA, lda), (1, n, dB, ldb)):
            op = torch.empty(oz.oz_operand_bytes(s, ln, k, sid, rt), dtype=torch.uint8, device="cuda")
            before = oz.oz_launch_count()
            oz.check(oz.oz_prepare_operand(s, ln, k, dX, ld, sid, rt, op), "oz_prepare_operand")
            launches.append(oz.oz_launch_count() - before)
            ops.append(op)
        assert launches[side] == 1
        dC = torch.zeros((n, m), dtype=torch.float64, device="cuda")
        oz.check(oz.oz_dgemm_prepared(m, n, k, 1.0, *ops, 0.0, dC, m, sid, rt), "oz_dgemm_prepared")
        assert oz.oz_query_status() == oz.OZ_ERR_NONFINITE_INPUT
        _same(gh.from_dev(dC), ozo.dgemm(A, B, OSET[set_name], getattr(ozo, "QUANT_" + quant), getattr(ozo, "SCALE_" + rule)))


@pytest.mark.parametrize("set_name,sub", ROUTES)
@pytest.mark.parametrize("m,n,k,pad", [(4699, 33, 1191, 1), (2970, 140, 1893, 0), (36, 4700, 1190, 0), (140, 1785, 3149, 0)])
def test_row_check(m, n, k, pad, set_name, sub):
    """The row check on the scan results that the form leaves: whole calls (with the two-plane layouts of A where n <= 128)."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + n + k)
    # rows of A from flat to wide; columns of B flat (less so for the larger set), since the widest of them counts for every row
    bs = 1.2 if set_name == "A" else 0.0
    A = _lines(rng, m, k, 3.5) if m > n else rng.standard_normal((m, k)) * np.exp(3.5 * rng.random((m, 1)) * rng.standard_normal((m, k)))
    B = rng.standard_normal((n, k)) * np.exp(bs * rng.standard_normal((n, k))) if m > n else _lines(rng, n, k, bs, spikes=False)
    A, B = np.asfortranarray(A), np.asfortranarray(B.T)
    C0 = np.asfortranarray(rng.standard_normal((m, n)))
    sid, rt = gh.SETS[set_name], gh.route(sub, fallback=True)
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, sid, rt))
    (dA, lda), (dB, ldb), dC = _device(A, pad, 0), _device(B, pad, 0), gh.to_dev(C0)
    oz.oz_query_fallback_rows()
    before = oz.oz_launch_count()
    oz.check(oz.oz_dgemm_ex(m, n, k, -1.0, dA, lda, dB, ldb, 1.0, dC, m, sid, rt), "oz_dgemm_ex")
    # two deconstructions, the check, the residue products, the reconstruction, the native rows
    assert oz.oz_launch_count() - before == 6
    want, flag = ozo.dgemm_fallback(A, B, OSET[set_name], ozo.QUANT_RN, -1.0, 1.0, C0)
    assert oz.oz_query_status() == oz.OZ_ERR_NONFINITE_INPUT
    assert 0 < flag.sum() < m and oz.oz_query_fallback_rows() == int(flag.sum())
    _same(gh.from_dev(dC), want)


@pytest.mark.parametrize("rule,quant", [("CS", "TZ"), ("MAXEXP", "RN")])
@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("E", "int8"), ("A", "int8n")])
def test_two_large_operands(set_name, sub, rule, quant):
    """Both operands by clusters, on two streams: sampled rows and columns of one product."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    m, n, k = 4699, 4701, 1191
    rng = np.random.default_rng(11)
    A, B = np.asfortranarray(_lines(rng, m, k)), np.asfortranarray(_lines(rng, n, k).T)
    got, st = gh.dgemm(A, B, set_name, gh.route(sub, quant, rule))
    assert st == oz.OZ_ERR_NONFINITE_INPUT
    rows = np.r_[0:12, m - 12:m, rng.integers(0, m, 8)]
    cols = np.r_[0:12, n - 12:n, rng.integers(0, n, 8)]
    want = ozo.dgemm(np.asfortranarray(A[rows]), np.asfortranarray(B[:, cols]), OSET[set_name], getattr(ozo, "QUANT_" + quant), getattr(ozo, "SCALE_" + rule))
    _same(got[np.ix_(rows, cols)], want)
