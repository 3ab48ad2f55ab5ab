"""The conversion's FP32 limb arithmetic where it can go wrong: quantised values at the edges of every
limb (bits 0, 16, 31, 45) and at the largest magnitude of the scale rule, planes bit for bit against the
oracle, from the one-kernel form and from the large-operand kernels, at ragged sizes and odd strides."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oz_oracle as ozo

pytestmark = pytest.mark.gpu

OSET = {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}
OSUB = {"fp8": ozo.SUB_FP8, "int8": ozo.SUB_INT8, "int8n": ozo.SUB_INT8_NATIVE}


def _limb_edges(rng, lines, k, side, t):
    """Every line holds +-(1 - 2^-53), so that MAXEXP with a budget of t bits scales by 2^t; the other entries are
    sums of up to three +-2^(b - t), b around the limb boundaries, and single bits anywhere in the range."""
    b = rng.choice([0, 1, 14, 15, 16, 17, 29, 30, 31, 32, 43, 44, 45, 46], size=(lines, k, 3))
    X = (rng.choice([-1.0, 0.0, 1.0], size=b.shape) * np.exp2(b - float(t))).sum(axis=2)
    X += rng.choice([0.0, 0.0, 1.0, -1.0], size=(lines, k)) * np.exp2(-rng.integers(1, t, size=(lines, k)).astype(float))
    X = np.clip(X, -0.75, 0.75)
    X[np.arange(lines), rng.integers(0, k, size=lines)] = rng.choice([1.0, -1.0], size=lines) * (1.0 - 2.0 ** -53)
    X = X * np.exp2(rng.integers(-300, 300, size=lines).astype(float))[:, None]
    return np.asfortranarray(X if side == 0 else X.T)


@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("S", "int8"), ("E", "fp8"), ("E", "int8"), ("A", "fp8"),
                                          ("A", "int8"), ("A", "int8n")])
@pytest.mark.parametrize("side,lines,k", [(0, 37, 131), (1, 37, 131), (0, 1, 1), (0, 2101, 2051), (1, 2101, 2051),
                                          (1, 33, 131100)])
def test_limb_edges_bit_exact(side, lines, k, set_name, sub):
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(1000 * lines + k + side)
    t = ozo.budget_maxexp(OSET[set_name], k)[side]
    X = _limb_edges(rng, lines, k, side, t)
    for rule, quant in (("MAXEXP", "RN"), ("CS", "TZ")):
        got, shift, st = gh.deconstruct(side, X, set_name, gh.route(sub, quant, rule))
        want_shift = ozo.shifts(side, X, OSET[set_name], getattr(ozo, "SCALE_" + rule), t)
        Q = ozo.quantise(side, X, want_shift, getattr(ozo, "QUANT_" + quant))
        want = ozo.planes(ozo.residues(Q, OSET[set_name]), OSET[set_name], OSUB[sub])
        assert st == 0 and (shift == want_shift).all()
        assert got.shape == want.shape and (got == want).all()


@pytest.mark.parametrize("m,n,k", [
    (1, 1, 1), (3, 2, 5),            # less than one group of lines
    (9, 300, 64), (300, 9, 64),      # very unequal shares of the resident blocks
    (517, 403, 260),                 # groups of four lines on side 0, ragged
    (1301, 299, 1400),               # one large block per SM
    (1500, 1490, 1500),              # more rounds than one: two streams
    (150, 2100, 2051),               # one operand too large for the one-kernel form
])
@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("A", "int8n")])
def test_joint_deconstruction_shapes(m, n, k, set_name, sub):
    """Whole calls on either side of every rule that decides how the two operands are deconstructed together,
    against the call on operands that were prepared one by one (bit for bit: same shifts, same planes)."""
    import paper_2609_09095_b200 as oz
    import torch
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + 3 * n + k)
    A, B = np.asfortranarray(rng.standard_normal((m, k))), np.asfortranarray(rng.standard_normal((k, n)))
    A[0, 0] = 0.0
    if m > 8:
        A[5, :] = 0.0
        A[7, :] *= 2.0 ** -1060                       # a row of subnormals
    if n > 4:
        B[:, 3] *= 2.0 ** 700
    got, st = gh.dgemm(A, B, set_name, gh.route(sub))
    rt, S = gh.route(sub), gh.SETS[set_name]
    opA = torch.empty(oz.oz_operand_bytes(0, m, k, S, rt), dtype=torch.uint8, device="cuda")
    opB = torch.empty(oz.oz_operand_bytes(1, n, k, S, rt), dtype=torch.uint8, device="cuda")
    oz.check(oz.oz_prepare_operand(0, m, k, gh.to_dev(A), m, S, rt, opA), "prepare A")
    oz.check(oz.oz_prepare_operand(1, n, k, gh.to_dev(B), k, S, rt, opB), "prepare B")
    dC = torch.full((n, m), 7.0, dtype=torch.float64, device="cuda")
    oz.check(oz.oz_dgemm_prepared(m, n, k, 1.0, opA, opB, 0.0, dC, m, S, rt), "product")
    assert st == 0 and gh.sync_status() == 0
    assert (got == gh.from_dev(dC)).all()
    if m * n <= 200000:
        assert (got == ozo.dgemm(A, B, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS)).all()


@pytest.mark.parametrize("lines,k", [
    (42001, 100),               # one piece of a line per row of a conversion tile
    (33001, 130),               # two, the second one cut off by the row pitch
    (703, 6001),                # 47 pieces a line: tiles start in the middle of lines, the last one is partly empty
    (3, 33000),                 # fewer rows than resident tiles
])
@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("E", "int8"), ("A", "int8n")])
def test_three_pass_deconstruction_of_columns(lines, k, set_name, sub):
    """Columns too long or too many for the one-kernel form, planes in the documented layout: sampled lines are the
    oracle's, and all bytes are those of the same columns deconstructed a few at a time."""
    import torch
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(lines + k)
    X = np.asfortranarray(rng.standard_normal((k, lines)))
    X[:, lines // 2] = 0.0
    X[k // 2, 1] = np.inf
    rt = gh.route(sub)
    got, shift, st = gh.deconstruct(1, X, set_name, rt)
    assert st != 0 and shift[1] == -2 ** 31 and (got[:, 1] == 0).all()
    pick = np.unique(np.array([0, 2 % lines, lines // 3, lines // 2, max(lines - 2, 0), lines - 1]))
    pick = pick[pick != 1]
    Y = np.asfortranarray(X[:, pick])
    want_shift = ozo.shifts(1, Y, OSET[set_name], ozo.SCALE_CS, 0)
    Q = ozo.quantise(1, Y, want_shift, ozo.QUANT_RN)
    D = ozo.residues(Q, OSET[set_name])
    assert (shift[pick] == want_shift).all()
    assert (got[:, pick] == ozo.planes(D, OSET[set_name], OSUB[sub])).all()
    step = max(1, min(lines, 2 ** 20 // k))
    for a in range(0, lines, step):
        part, part_shift, _ = gh.deconstruct(1, np.asfortranarray(X[:, a:a + step]), set_name, rt)
        assert (shift[a:a + step] == part_shift).all() and (got[:, a:a + step] == part).all()


@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("E", "int8"), ("A", "int8n")])
@pytest.mark.parametrize("m,n,k", [(1003, 301, 5003), (33, 2049, 8193), (2600, 9, 4097),
                                   (450, 640, 9601)])            # both operands in three passes, in one launch each
def test_scan_by_guessed_exponents(set_name, sub, m, n, k):
    """The scan of large operands guesses a line's largest exponent from a sample: lines whose largest element hides between the samples,
    by no, one, two, three and many powers of two, lines of zeros, of subnormals, with samples of zeros only, with Inf and NaN, and lines whose
    samples spread so far that there is no guess."""
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + n + k)
    A, B = np.asfortranarray(rng.standard_normal((m, k))), np.asfortranarray(rng.standard_normal((k, n)))
    hidden = k // 32 + 5                              # no sample: samples lie at the multiples of k / 32, or four behind each of k / 8
    for lines, axis in ((A, 0), (B, 1)):
        count = lines.shape[axis]
        rows = lines if axis == 0 else lines.T
        for i, e in zip(range(count), (0, 1, 2, 3, 4, 60, -30, 900)):
            rows[i] = np.clip(rows[i], -1.9, 1.9)
            rows[i, hidden] = 1.5 * 2.0 ** e
        if count > 20:
            rows[9], rows[10] = 0.0, rows[10] * 2.0 ** -1060
            rows[11, hidden + 1:], rows[11, :hidden] = 0.0, 0.0
            rows[12] *= 2.0 ** -1000
            rows[13] *= 2.0 ** 900
            for sample in [i * k // 32 for i in range(32)] + [i * k // 8 + u for i in range(8) for u in range(4)]:
                rows[14, sample] = 0.0
            rows[15, hidden] = 5e-324
            rows[16, 0] = 2.0 ** 300
            rows[17] *= np.exp(3.0 * rng.standard_normal(k))
            rows[18] *= np.exp(1.2 * rng.standard_normal(k))
        if count > 200:
            rows[96:128] *= np.exp(2.0 * rng.standard_normal((32, k)))
    if m > 100:
        A[20, 5], A[21, hidden] = np.nan, np.inf
    rt = gh.route(sub)
    got, _ = gh.dgemm(A, B, set_name, rt)
    want = ozo.dgemm(A, B, {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}[set_name], ozo.QUANT_RN, ozo.SCALE_CS)
    assert (np.isnan(got) == np.isnan(want)).all()
    assert (got[~np.isnan(want)] == want[~np.isnan(want)]).all()
