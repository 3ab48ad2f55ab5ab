"""oz_dgemm_host panel by panel: shapes around the rules that cut a call into column panels, every form of a
call that takes or declines them, bit for bit against the device-pointer entry point."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k,alpha,beta,set_name,sub,rule,recon", [
    (300, 511, 90, 1.0, 0.0, "S", "fp8", "CS", None),          # too few columns for whole-tile panels
    (1500, 512, 200, -1.0, 1.0, "S", "fp8", "CS", None),       # two panels of one tile
    (1500, 513, 200, -1.0, 1.0, "S", "int8", "MAXEXP", None),  # a column beyond whole tiles
    (777, 2003, 1021, 1.0, 0.0, "E", "fp8", "CS", None),       # ragged panels, B wider than C
    (40, 5003, 700, 1.0, 1.0, "A", "int8n", "CS", None),       # few rows: the traffic is B's
    (2500, 300, 260, -1.0, 1.0, "S", "fp8", "CS", None),       # C in panels, the product undivided
    (1200, 1300, 400, 1.0, 1.0, "S", "fp8", "ACCURATE", None), # shifts of A from all of B: product undivided
    (1200, 1300, 400, -1.0, 1.0, "S", "fp8", "CS", "tensor"),
])
def test_host_panels_bit_identical(m, n, k, alpha, beta, set_name, sub, rule, recon):
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + n + k)
    A, B = np.asfortranarray(rng.standard_normal((m, k))), np.asfortranarray(rng.standard_normal((k, n)))
    B[:, n - 1] = 0.0
    A[m // 2, 0] = np.nan                                # a row of NaN in every panel
    C0 = np.asfortranarray(rng.standard_normal((m, n)))
    lda, ldb, ldc = m + 1, k + 3, m + 2
    host = lambda X, ld: torch.from_numpy(np.ascontiguousarray(np.vstack([X, np.full((ld - X.shape[0], X.shape[1]), 5.0)]).T)).pin_memory()
    hA, hB, hC = host(A, lda), host(B, ldb), host(C0, ldc)
    rt, S = gh.route(sub, "RN", rule, recon=recon), gh.SETS[set_name]
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, S, rt) + 8 * (m * k + k * n + m * n) + 1024)
    want, st = gh.dgemm(A, B, set_name, rt, alpha, beta, C0 if beta else None)
    for _ in range(2):
        hC.copy_(host(C0, ldc))
        oz.check(oz.oz_dgemm_host(m, n, k, alpha, hA, lda, hB, ldb, beta, hC, ldc, S, rt), "oz_dgemm_host")
        assert gh.sync_status() == st == oz.OZ_ERR_NONFINITE_INPUT
        got = hC.numpy().T
        assert (got[m:] == 5.0).all()
        np.testing.assert_array_equal(got[:m], want)


def test_host_routes_taken_undivided():
    """Row check and storage mode F stay accepted at sizes that other calls cut into panels."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(3)
    for m, n, k, extra in ((1500, 1400, 64, oz.OZ_FALLBACK_FP64), (12000, 128, 256, oz.OZ_STORAGE_FUSED)):
        A, B = np.asfortranarray(rng.standard_normal((m, k))), np.asfortranarray(rng.standard_normal((k, n)))
        rt, S = gh.route("fp8") | extra, oz.OZ_SET_S
        gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, S, rt) + 8 * (m * k + k * n + m * n) + 1024)
        hA, hB = (torch.from_numpy(np.ascontiguousarray(X.T)).pin_memory() for X in (A, B))
        hC = torch.zeros((n, m), dtype=torch.float64).pin_memory()
        oz.check(oz.oz_dgemm_host(m, n, k, 1.0, hA, m, hB, k, 0.0, hC, m, S, rt), "oz_dgemm_host")
        want, st = gh.dgemm(A, B, "S", gh.route("fp8"))
        assert gh.sync_status() == st == 0
        assert (hC.numpy().T == want).all()


def test_refused_call_leaves_nothing_behind():
    """A host call that is refused enqueues no copy: the device call that follows at once in the same workspace has its
    planes and residues to itself."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(8)
    m, n, k, S = 1500, 1400, 64, oz.OZ_SET_S
    rt, accurate = gh.route("fp8"), gh.route("fp8", "RN", "ACCURATE")
    hA, hB, hC = (torch.full(shape, 3.0, dtype=torch.float64).pin_memory() for shape in ((k, m), (n, k), (n, m)))
    A, B = np.asfortranarray(rng.standard_normal((m, 900))), np.asfortranarray(rng.standard_normal((900, n)))
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, 900, S, rt) + 8 * (m * k + k * n + m * n) + 1024)
    want, _ = gh.dgemm(A, B, "S", rt)
    dA, dB, dC = gh.to_dev(A), gh.to_dev(B), torch.zeros((n, m), dtype=torch.float64, device="cuda")
    for _ in range(4):
        before = oz.oz_launch_count()
        assert oz.oz_dgemm_host(m, n, k, 2.0, hA, m, hB, k, 1.0, hC, m, S, rt) == oz.OZ_ERR_UNSUPPORTED
        assert oz.oz_dgemm_host(m, n, 16385, 1.0, hA, m, hB, 16385, 1.0, hC, m, S, accurate) == oz.OZ_ERR_UNSUPPORTED
        assert oz.oz_launch_count() == before
        oz.check(oz.oz_dgemm_ex(m, n, 900, 1.0, dA, m, dB, 900, 0.0, dC, m, S, rt), "oz_dgemm_ex")
    assert gh.sync_status() == 0
    assert (gh.from_dev(dC) == want).all() and bool((hC == 3.0).all())


@pytest.mark.parametrize("which", ["ABC", "B", "C"])
def test_pageable_buffers_are_not_cut_up(which):
    """Copies of pageable memory overlap nothing: such a call is the device call between its copies, kernel for kernel."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(12)
    m, n, k, S, rt = 1500, 1401, 300, oz.OZ_SET_S, gh.route("fp8")
    A, B, C0 = (np.asfortranarray(rng.standard_normal(shape)) for shape in ((m, k), (k, n), (m, n)))
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, S, rt) + 8 * (m * k + k * n + m * n) + 1024)
    host = {name: torch.from_numpy(np.ascontiguousarray(X.T)) for name, X in (("A", A), ("B", B), ("C", C0))}
    host = {name: t if name in which else t.pin_memory() for name, t in host.items()}
    before = oz.oz_launch_count()
    want, st = gh.dgemm(A, B, "S", rt, -1.0, 1.0, C0)
    undivided = oz.oz_launch_count() - before
    oz.check(oz.oz_dgemm_host(m, n, k, -1.0, host["A"], m, host["B"], k, 1.0, host["C"], m, S, rt), "oz_dgemm_host")
    assert gh.sync_status() == st == 0
    assert oz.oz_launch_count() - before == 2 * undivided
    assert (host["C"].numpy().T == want).all()
