"""Two-plane schedule of products with at most 128 columns: d = d0 + 16 d1 of a non-square modulus meets e and 16 e (planes
private to a call) or e with the second plane negated (planes of kept operands).  Bit for bit the oracle's result at the edges
of its tiles and of the exact depths of its accumulators."""
import numpy as np
import pytest

import synth_inputs as syn
from oracle import oz_oracle as ozo

pytestmark = pytest.mark.gpu

OSET = {"S": ozo.SET_S, "E": ozo.SET_E, "A": ozo.SET_A}


@pytest.mark.parametrize("set_name", ["S", "E", "A"])
@pytest.mark.parametrize("sub", ["fp8", "int8"])
@pytest.mark.parametrize("m,n,k,quant,rule", [(1, 1, 1, "RN", "CS"), (128, 128, 128, "TZ", "CS"), (255, 100, 129, "RN", "MAXEXP"),
                                              (257, 127, 1000, "RN", "CS"), (600, 8, 4101, "RN", "ACCURATE"), (2500, 33, 2049, "RN", "CS")])
def test_whole_method(set_name, sub, m, n, k, quant, rule):
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + 3 * n + 5 * k)
    A, B = syn._draw(rng, m, k, "lognormal:0.5"), syn._draw(rng, k, n, "normal")
    if m > 4:
        A[3, :] = 0.0
        A[2, k // 2] = 1e9
    C0 = np.asfortranarray(rng.standard_normal((m, n)))
    got, st = gh.dgemm(A, B, set_name, gh.route(sub, quant, rule), -1.0, 1.0, C0)
    assert st in (0, 6)             # 6: the exponent-span check on the spike
    want = ozo.dgemm(A, B, OSET[set_name], getattr(ozo, f"QUANT_{quant}"), getattr(ozo, f"SCALE_{rule}"), -1.0, 1.0, C0)
    assert (got == want).all()


@pytest.mark.parametrize("set_name", ["S", "E", "A"])
@pytest.mark.parametrize("m,n,k", [(300, 100, 3840), (300, 16, 3841), (130, 128, 15361), (40, 8, 33000)])
def test_depth_with_like_signs(set_name, m, n, k):
    """Constant lines: every product has the same sign, so the accumulators come close to their bounds.  The kept operands
    carry -16 d1 and are cut into K segments from 3840 (S) or 15360 (E, A), the whole call from 32768."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + k)
    A = np.asfortranarray(np.broadcast_to(rng.uniform(0.5, 2.0, size=(m, 1)), (m, k)))
    B = np.asfortranarray(np.broadcast_to(rng.uniform(-2.0, -0.5, size=(1, n)), (k, n)))
    A[: m // 2] = syn._draw(rng, m // 2, k, "uniform")
    want = ozo.dgemm(A, B, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS)
    sid, rt = gh.SETS[set_name], gh.route("fp8")
    got, st = gh.dgemm(A, B, set_name, rt)
    assert st == 0 and (got == want).all()
    ops = [torch.empty(oz.oz_operand_bytes(side, lines, k, sid, rt), dtype=torch.uint8, device="cuda") for side, lines in ((0, m), (1, n))]
    oz.check(oz.oz_prepare_operand(0, m, k, gh.to_dev(A), m, sid, rt, ops[0]), "oz_prepare_operand A")
    oz.check(oz.oz_prepare_operand(1, n, k, gh.to_dev(B), k, sid, rt, ops[1]), "oz_prepare_operand B")
    gh.ensure_workspace(oz.oz_product_workspace_bytes(m, n, sid))
    dC = torch.zeros((n, m), dtype=torch.float64, device="cuda")
    oz.check(oz.oz_dgemm_prepared(m, n, k, 1.0, *ops, 0.0, dC, m, sid, rt), "oz_dgemm_prepared")
    assert gh.sync_status() == 0 and (gh.from_dev(dC) == want).all()


@pytest.mark.parametrize("sub", ["fp8", "int8"])
@pytest.mark.parametrize("m,n,k", [(40, 1, 33), (200, 31, 300), (300, 32, 129), (2000, 33, 260), (700, 63, 1000), (9600, 64, 130), (500, 64, 4300)])
def test_stacked_accumulators(sub, m, n, k):
    """At most 64 columns: both accumulators of a modulus from one chain, handed from one half of the epilogue to the other.  Edges of the
    warps' 32 columns, tiles of 64 and of 256 rows, several products a block and several K segments; whole calls and kept operands."""
    import torch
    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    rng = np.random.default_rng(m + n + k)
    A, B = syn._draw(rng, m, k, "normal"), syn._draw(rng, k, n, "lognormal:0.5")
    rt = gh.route(sub)
    for set_name, sid in gh.SETS.items():
        want = ozo.dgemm(A, B, OSET[set_name], ozo.QUANT_RN, ozo.SCALE_CS)
        got, st = gh.dgemm(A, B, set_name, rt)
        assert st == 0 and (got == want).all()
        block = [torch.empty(oz.oz_operand_bytes(side, lines, k, sid, rt), dtype=torch.uint8, device="cuda") for side, lines in ((0, m), (1, n))]
        oz.check(oz.oz_prepare_operand(0, m, k, gh.to_dev(A), m, sid, rt, block[0]), "oz_prepare_operand A")
        oz.check(oz.oz_prepare_operand(1, n, k, gh.to_dev(B), k, sid, rt, block[1]), "oz_prepare_operand B")
        gh.ensure_workspace(oz.oz_product_workspace_bytes(m, n, sid))
        dC = gh.to_dev(np.zeros((m, n), order="F"))
        oz.check(oz.oz_dgemm_prepared(m, n, k, 1.0, *block, 0.0, dC, m, sid, rt), "oz_dgemm_prepared")
        assert gh.sync_status() == 0 and (gh.from_dev(dC) == want).all()
