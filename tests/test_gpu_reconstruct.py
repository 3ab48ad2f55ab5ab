"""Reconstruction at the edges of its fast path: scales whose power of two is no normal double, integers next to a
rounding boundary, to a power of two and to +-M/2, marked lines.  The same values against every shift."""
import numpy as np
import pytest

from oracle import oz_oracle as ozo

pytestmark = pytest.mark.gpu

OSET = {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}
MARK = -(2 ** 31)


@pytest.mark.parametrize("set_name", ["S", "E", "A"])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.0, 1.0)])
def test_scale_and_rounding_edges(set_name, alpha, beta):
    import tests.gpu_helpers as gh
    ms = ozo.modset(OSET[set_name])
    M = int(np.prod([int(v) for v in ms], dtype=object))
    xs = [0, 1, -1, 3, M // 2 - 1, -(M // 2), M // 2 - 2 ** 60, (M >> 1) - (M >> 22), -(M >> 1) + (M >> 31)]
    for e in (53, 54, 60, 77, 81, 95, 106, 109):
        tie_below, tie_above = 2 ** e - 2 ** max(e - 54, 0), 2 ** e + 2 ** max(e - 53, 0)
        xs += [2 ** e, tie_below, tie_below + 1, tie_below - 1, -tie_above, tie_above + 1, -(tie_above - 1)]
    # a rounding error just inside and just outside the guard of 2^-29 half units in the last place
    xs += [2 ** 105 + 2 ** 52 - 2 ** 22, 2 ** 105 + 2 ** 52 - 2 ** 24, -(2 ** 105 + 2 ** 53 + 2 ** 52 + 2 ** 24)]
    shifts = [-1200, -1010, -905, -904, -903, -100, 0, 57, 1019, 1020, 1021, 1022, 1100, 1180, MARK]
    m, n = len(xs), len(shifts)
    R = np.empty((len(ms), n, m), dtype=np.uint16)
    for i, mm in enumerate(ms):
        R[i] = np.array([x % mm for x in xs], dtype=np.uint16)
    sA = np.zeros(m, dtype=np.int32)
    sA[-1] = MARK                                    # a marked row against every column, the marked one among them
    sB = np.array(shifts, dtype=np.int32)
    C0 = np.asfortranarray(np.random.default_rng(7).standard_normal((m, n)))
    CI = ozo.crt(R, OSET[set_name])
    for ldr, rows in ((None, m), (None, m - 1)):     # pairs of rows whole, and a last row alone
        Rr, CIr = np.ascontiguousarray(R[:, :, m - rows:]), CI[:, m - rows:]
        got, _ = gh.reconstruct(Rr, sA[m - rows:], sB, set_name, alpha, beta, C0[m - rows:], ldr=ldr)
        want = ozo.output(np.ascontiguousarray(CIr), sA[m - rows:], sB, alpha, beta, np.asfortranarray(C0[m - rows:]))
        assert (np.isnan(got) == np.isnan(want)).all()
        assert (got[~np.isnan(want)] == want[~np.isnan(want)]).all()


@pytest.mark.parametrize("set_name", ["S", "E", "A"])
def test_marks_and_far_shifts(set_name):
    """A marked line gives NaN whatever the shift of its partner, and shifts whose sum leaves 32 bits give zero or infinity
    like any other sum that far out."""
    import tests.gpu_helpers as gh
    ms = ozo.modset(OSET[set_name])
    top = 2 ** 31 - 1
    sA = np.array([MARK, -(2 ** 29) - 904, -(2 ** 29), -(2 ** 29) + 57, -(2 ** 29) + 1020, 2 ** 29 + 57, 2 ** 30, 2 ** 30 + 1, -(2 ** 30) - 1,
                   top, top - 56, -top, -top + 57, 0, 57], dtype=np.int32)
    sB = np.array([MARK, 0, 57, top, top - 904, top - 2 ** 29, -top, -top + 57, -top + 1020, -(2 ** 30) - 5, 2 ** 29, 3 - 2 ** 29], dtype=np.int32)
    m, n = len(sA), len(sB)
    xs = np.array([[(-1) ** (i + j) * (3 + i + 16 * j) for i in range(m)] for j in range(n)], dtype=object)
    R = np.array([[[x % int(mm) for x in row] for row in xs] for mm in ms], dtype=np.uint16)
    got, _ = gh.reconstruct(R, sA, sB, set_name)
    for i in range(m):
        for j in range(n):
            s = int(sA[i]) + int(sB[j])
            if MARK in (int(sA[i]), int(sB[j])):
                assert np.isnan(got[i, j]), (int(sA[i]), int(sB[j]))
            else:
                sign = -1.0 if xs[j][i] < 0 else 1.0
                want = sign * np.inf if s < -2000 else 0.0 if s > 2000 else float(xs[j][i]) * 2.0 ** -s if s < 1000 else np.ldexp(float(xs[j][i]), -s)
                assert got[i, j] == want, (int(sA[i]), int(sB[j]))


@pytest.mark.parametrize("set_name,sub,recon", [("S", "fp8", None), ("S", "int8", None), ("E", "fp8", None), ("E", "int8", None), ("A", "fp8", None),
                                                ("A", "int8", None), ("A", "int8n", None), ("S", "fp8", "tensor"), ("E", "int8", "tensor")])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (63, 31, 5), (64, 32, 40), (65, 33, 64), (80, 129, 17), (257, 65, 96), (1200, 1090, 33)])
def test_stored_forms_and_small_results(set_name, sub, recon, m, n, k):
    """Residues of every stored form through edges of patches (32 columns x 64 rows, chunks of sixteen) and more patches than the blocks of a round:
    outputs that are zero, that cancel almost to nothing, whose integers span the range of a row, and ordinary ones."""
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m * 7 + n * 3 + k)
    A = rng.standard_normal((m, k))
    B = rng.standard_normal((k, n))
    A[::5, : k // 2] = 0.0                            # rows and columns that share no index: products that are zero
    B[k // 2:, ::3] = 0.0
    A[::7] = np.round(A[::7] * 4.0)                   # integers, many results equal or zero
    if k > 1:
        A[1::11, 1] = A[1::11, 0]                     # cancels to 2^-40 of the terms
        B[1, 1::6] = -B[0, 1::6] * (1.0 + 2.0 ** -40)
        A[1::11, 2:] = 0.0
    B[:, 2::13] *= 2.0 ** rng.integers(-70, 1, size=B[:, 2::13].shape).astype(np.float64)
    for alpha, beta, pad in ((1.0, 0.0, 0), (-1.0, 1.0, 0), (-1.0, 1.0, 1), (-1.0, 0.0, 1)):
        C0 = np.asfortranarray(rng.standard_normal((m, n)))
        rt = gh.route(sub, recon=recon)
        gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, gh.SETS[set_name], rt))
        Af, Bf = np.asfortranarray(A), np.asfortranarray(B)
        Cp = np.asfortranarray(np.vstack([C0, np.full((pad + m % 2, n), 3.0)]))       # even and odd leading dimensions
        dC = gh.to_dev(Cp)
        oz.check(oz.oz_dgemm_ex(m, n, k, alpha, gh.to_dev(Af), m, gh.to_dev(Bf), k, beta, dC, Cp.shape[0], gh.SETS[set_name], rt), "oz_dgemm_ex")
        assert gh.sync_status() == 0
        got = gh.from_dev(dC)
        want = ozo.dgemm(Af, Bf, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS, alpha=alpha, beta=beta, C0=C0)
        assert (got[:m] == want).all() and (got[m:] == 3.0).all()


@pytest.mark.parametrize("set_name", ["S", "E", "A"])
@pytest.mark.parametrize("ldr", [None, 1024, 1025])
def test_integers_of_every_magnitude(set_name, ldr):
    """c' of every bit length up to M/2: a power of two and its neighbours, the ties of every length above 53 bits and theirs, random ones; four
    shifts each, so that rows that the floating sum settles lie beside rows that it leaves open."""
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(11)
    ms = ozo.modset(OSET[set_name])
    M = int(np.prod([int(v) for v in ms], dtype=object))
    xs = [0]
    for e in range(M.bit_length() - 1):
        tie = 2 ** e + 2 ** max(e - 53, 0)
        x = 2 ** e + int(rng.integers(0, 2 ** 62)) * 2 ** max(e - 62, 0) % 2 ** e + int(rng.integers(0, 2 ** 40)) % 2 ** min(e, 40)
        xs += [s * v for s in (1, -1) for v in (2 ** e, 2 ** e - 1, tie, tie - 1, tie + 1, x)]
    xs = [x for x in xs if -(M // 2) <= x < M // 2]
    m = 1023 if ldr else len(xs)
    xs = (xs * 2)[:m]
    sB = np.array([0, 57, -900, 900], dtype=np.int32)
    row = np.array([[x % int(mm) for x in xs] for mm in ms], dtype=np.uint16)
    R = np.ascontiguousarray(np.broadcast_to(row[:, None, :], (len(ms), 4, m)))
    R[:, 1] = R[:, 1, rng.permutation(m)]                                             # small ones next to large ones
    sA = np.zeros(m, dtype=np.int32)
    C0 = np.asfortranarray(rng.standard_normal((m, 4)))
    for alpha, beta in ((1.0, 0.0), (-1.0, 1.0)):
        got, _ = gh.reconstruct(R, sA, sB, set_name, alpha, beta, C0, ldr=ldr)
        assert (got == ozo.output(ozo.crt(R, OSET[set_name]), sA, sB, alpha, beta, C0)).all()


@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("E", "int8"), ("A", "int8n")])
@pytest.mark.parametrize("m,n", [(200, 300), (1001, 900)])
@pytest.mark.parametrize("fall", [2.0, 5.0, 20.0])
def test_graded_operands(set_name, sub, m, n, fall):
    """Whole calls on operands that fall off from the diagonal: results of every size below the bound of their row and column, two rows a
    thread and four."""
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + int(fall))
    k = 150
    away = lambda p, q: np.exp(-np.abs(np.arange(p)[:, None] * (q / p) - np.arange(q)[None, :]) / fall)     # noqa: E731
    A, B = np.asfortranarray(rng.standard_normal((m, k)) * away(m, k)), np.asfortranarray(rng.standard_normal((k, n)) * away(k, n))
    C0 = np.asfortranarray(rng.standard_normal((m, n)) * 1e-9)
    for alpha, beta in ((1.0, 0.0), (-1.0, 1.0)):
        got, st = gh.dgemm(A, B, set_name, gh.route(sub), alpha, beta, C0)
        assert st == 0 and (got == ozo.dgemm(A, B, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS, alpha=alpha, beta=beta, C0=C0)).all()


@pytest.mark.parametrize("set_name,sub,recon", [("S", "fp8", None), ("E", "int8", None), ("A", "int8n", None), ("S", "fp8", "tensor"), ("A", "int8n", "tensor")])
@pytest.mark.parametrize("m,pad", [(64, 0), (75, 0), (75, 1), (1003, 0), (1002, 1)])
def test_zeros_are_positive(set_name, sub, recon, m, pad):
    """C = - A B without an old value: results that are zero, or too small and negative, are +0 in whatever group of rows and form of store they lie."""
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + pad)
    n, k = 800, 40
    A, B = np.asfortranarray(rng.standard_normal((m, k))), np.asfortranarray(rng.standard_normal((k, n)))
    A[::3, : k // 2], B[k // 2:, ::2] = 0.0, 0.0
    A[1::6] *= 2.0 ** -1000
    B[:, 1::4] *= 2.0 ** -900
    rt = gh.route(sub, recon=recon)
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, gh.SETS[set_name], rt))
    dC = gh.to_dev(np.asfortranarray(np.full((m + pad, n), 3.0)))
    oz.check(oz.oz_dgemm_ex(m, n, k, -1.0, gh.to_dev(A), m, gh.to_dev(B), k, 0.0, dC, m + pad, gh.SETS[set_name], rt), "oz_dgemm_ex")
    assert gh.sync_status() == 0
    got = gh.from_dev(dC)[:m]
    assert (got == 0.0).mean() > 0.2 and not np.signbit(got[got == 0.0]).any()
