"""Calls that follow one another without a synchronisation, host-buffer calls inside a stream capture, and operand
entries beyond the exact range of the conversion."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oz_oracle as ozo

pytestmark = pytest.mark.gpu

OSET = {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}


def test_calls_back_to_back_in_one_workspace():
    """Calls of different shapes and routes enqueued one behind the other: every kernel is launched as a dependent of
    its predecessor and may start early, so one that does not wait reads (or overwrites) the workspace of the call before.
    Each output is that of the same call made alone, bit for bit."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    gen = torch.Generator(device="cuda").manual_seed(5)
    jobs = []
    for m, n, k, set_name, sub, rule, extra in [
            (256, 256, 256, "S", "fp8", "CS", 0),                        # joint deconstruction, early reconstruction
            (1500, 1490, 1500, "S", "fp8", "CS", 0),                     # two streams, one-kernel form of each operand
            (200, 300, 260, "A", "int8n", "MAXEXP", 0),
            (3000, 2500, 1700, "E", "int8", "CS", 0),                    # three passes over both: joint scans, then two streams
            (1000, 900, 5003, "S", "fp8", "CS", 0),                      # the same with lines too long for a cluster
            (4700, 4500, 1190, "E", "int8", "CS", 0),                    # both by clusters, on two streams
            (4700, 64, 1190, "S", "fp8", "CS", oz.OZ_FALLBACK_FP64),     # A by clusters, with the row check behind it
            (64, 33, 700, "S", "int8", "CS", 0),
            (700, 650, 500, "S", "fp8", "ACCURATE", 0),
            (2000, 100, 900, "S", "fp8", "CS", oz.OZ_STORAGE_FUSED),
            (500, 450, 300, "S", "fp8", "CS", oz.OZ_FALLBACK_FP64),
            (300, 290, 5003, "S", "fp8", "CS", 0),                       # K segments
            (400, 300, 200, "S", "fp8", "CS", oz.OZ_RECON_TENSOR)]:
        new = lambda *shape: torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)
        jobs.append((m, n, k, gh.SETS[set_name], gh.route(sub, "RN", rule) | extra, new(k, m), new(n, k), new(n, m)))
    gh.ensure_workspace(max(oz.oz_workspace_bytes(*j[:3], j[3], j[4]) for j in jobs))

    def call(j, C):
        m, n, k, set_id, rt, A, B, _ = j
        oz.check(oz.oz_dgemm_ex(m, n, k, -1.0, A, m, B, k, 1.0, C, m, set_id, rt), "oz_dgemm_ex")

    alone = []
    for j in jobs:
        C = j[7].clone()
        call(j, C)
        torch.cuda.synchronize()
        alone.append(C)
    rng = np.random.default_rng(0)
    for _ in range(8):
        order = [int(i) for i in rng.integers(0, len(jobs), 30)]
        outs = [jobs[i][7].clone() for i in order]
        torch.cuda.synchronize()
        for i, C in zip(order, outs):
            call(jobs[i], C)
        torch.cuda.synchronize()
        assert gh.sync_status() == 0
        for i, C in zip(order, outs):
            assert torch.equal(C, alone[i]), jobs[i][:5]


@pytest.mark.parametrize("m,n,k,rule,alpha,beta", [
    (300, 280, 200, "CS", 1.0, 0.0),              # undivided: the copies are on the call's stream
    (1500, 1400, 64, "CS", -1.0, 1.0),            # product panel by panel
    (3000, 300, 260, "CS", -1.0, 1.0),            # C in panels, the product undivided
    (1200, 1300, 400, "ACCURATE", 1.0, 0.0),
])
def test_host_call_replayed_from_a_cuda_graph(m, n, k, rule, alpha, beta):
    """A host-buffer call captured after a plain one: the copy streams fork from and join the captured stream."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m)
    rt, S = gh.route("fp8", "RN", rule), oz.OZ_SET_S
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, S, rt) + 8 * (m * k + k * n + m * n) + 1024)
    hA, hB, hC = (torch.zeros(shape, dtype=torch.float64).pin_memory() for shape in ((k, m), (n, k), (n, m)))

    def call():
        oz.check(oz.oz_dgemm_host(m, n, k, alpha, hA, m, hB, k, beta, hC, m, S, rt, torch.cuda.current_stream()), "oz_dgemm_host")

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        call()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            call()
    for _ in range(3):
        A, B, C0 = (np.asfortranarray(rng.standard_normal(shape)) for shape in ((m, k), (k, n), (m, n)))
        for h, X in ((hA, A), (hB, B), (hC, C0)):
            h.copy_(torch.from_numpy(np.ascontiguousarray(X.T)))
        graph.replay()
        torch.cuda.synchronize()
        want, st = gh.dgemm(A, B, "S", rt, alpha, beta, C0 if beta else None)
        assert st == 0
        np.testing.assert_array_equal(hC.numpy().T, want)


@pytest.mark.parametrize("set_name,sub", [("S", "fp8"), ("S", "int8"), ("E", "fp8"), ("A", "fp8"), ("A", "int8n")])
def test_accurate_rule_entries_that_meet_only_zeros(set_name, sub):
    """Under the accurate rule an entry of A that only meets zeros of B may exceed the exact range of the conversion by
    far: its residues are arbitrary, index the digit table all the same, and add nothing to the product."""
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(17)
    m, n, k = 150, 140, 300
    A, B = np.asfortranarray(rng.standard_normal((m, k))), np.asfortranarray(rng.standard_normal((k, n)))
    dead = np.arange(0, k, 3)
    A[:, dead] *= 2.0 ** rng.integers(5, 40, (m, len(dead)))
    B[dead, :] = 0.0
    A[5, :] = 0.0
    A[5, dead] = rng.standard_normal(len(dead))           # a row that meets nothing but zeros
    B[1, :] *= 2.0 ** -20
    for i in (6, 70, 149):                                # rows whose bound product is as small as it can be
        A[i, :] = 0.0
        A[i, dead] = 2.0 ** 20 * rng.standard_normal(len(dead))
        A[i, 1] = rng.standard_normal()
    got, st = gh.dgemm(A, B, set_name, gh.route(sub, "RN", "ACCURATE"))
    assert st == 0
    # the same shifts with the dead entries left out: exact integer inner products of the live ones
    shA, shB, _, _ = ozo.shifts_accurate(A, B, OSET[set_name])
    live = np.setdiff1d(np.arange(k), dead)
    QA = ozo.quantise(0, np.asfortranarray(A[:, live]), shA, ozo.QUANT_RN)
    QB = ozo.quantise(1, np.asfortranarray(B[live, :]), shB, ozo.QUANT_RN)
    want = ozo.output(ozo.direct(QA, QB), shA, shB)
    np.testing.assert_array_equal(got, want)
    assert (got[5] == 0.0).all()
