"""What a call must not pay for: device times of the same work on other data or another leading dimension, as ratios.  The bounds
leave room above the ratios that the kernels show; the forms that they guard against lie above them."""
import pytest

pytestmark = pytest.mark.gpu

ROUTES = [("S", "fp8"), ("E", "fp8"), ("A", "int8n")]


def _ratio(slow, fast, tries=12):
    """Least device time of `slow` over that of `fast`, taken in turn."""
    import torch
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    best = [float("inf"), float("inf")]
    for t in range(tries + 2):
        for i, f in enumerate((slow, fast)):
            ev[0].record()
            for _ in range(3):
                f()
            ev[1].record()
            ev[1].synchronize()
            if t >= 2:
                best[i] = min(best[i], ev[0].elapsed_time(ev[1]))
    return best[0] / best[1]


def _normal(rows, cols, seed):
    import torch
    return torch.randn((cols, rows), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


def _residues(set_name, n, ldr, numbers, seed):
    """Random residues (numbers None), or those of whole numbers up to `numbers` in magnitude, for n columns of ldr rows."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    moduli = oz.oz_set_info(gh.SETS[set_name])[2]
    dt = gh.residue_dtype(set_name)[0]
    g = torch.Generator(device="cuda").manual_seed(seed)
    if numbers is None:
        return torch.stack([torch.randint(0, mm, (n, ldr), device="cuda", generator=g, dtype=torch.int32).to(dt) for mm in moduli])
    x = torch.randint(-numbers, numbers + 1, (n, ldr), device="cuda", generator=g, dtype=torch.int64)
    return torch.stack([(x % mm).to(torch.int32).to(dt) for mm in moduli])


@pytest.mark.parametrize("set_name,sub", ROUTES)
@pytest.mark.parametrize("numbers", [0, 2 ** 60])
def test_small_results_of_the_stage(set_name, sub, numbers):
    """Results that are zero or far below the bound of their row and column, by the public layout."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    m = n = 4000
    sA, sB = (torch.zeros(m, dtype=torch.int32, device="cuda") for _ in range(2))
    C = _normal(m, n, 1)
    calls = []
    for top in (numbers, None):
        R = _residues(set_name, n, m, top, 2)
        calls.append(lambda R=R: oz.check(oz.oz_reconstruct(m, n, R, m, n * m, sA, sB, gh.SETS[set_name], -1.0, 1.0, C, m)))
    assert _ratio(*calls) < (1.3 if numbers == 0 else 1.7)


@pytest.mark.parametrize("set_name,sub", ROUTES)
def test_small_results_of_a_product(set_name, sub):
    """One large entry in every row of A and column of B, so that nearly every result lies far below its bound."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    m = n = 4000
    k, rt = 128, gh.route(sub)
    gh.ensure_workspace(oz.oz_product_workspace_bytes(m, n, gh.SETS[set_name]))
    C = _normal(m, n, 1)
    calls = []
    for spike in (1e6, 1.0):
        A, B = _normal(m, k, 2), _normal(k, n, 3)
        A[torch.arange(m, device="cuda") % k, torch.arange(m, device="cuda")] *= spike
        B[torch.arange(n, device="cuda"), (torch.arange(n, device="cuda") * 7 + 3) % k] *= spike
        ops = [torch.empty(oz.oz_operand_bytes(s, m, k, gh.SETS[set_name], rt), dtype=torch.uint8, device="cuda") for s in (0, 1)]
        oz.check(oz.oz_prepare_operand(0, m, k, A, m, gh.SETS[set_name], rt, ops[0]))
        oz.check(oz.oz_prepare_operand(1, n, k, B, k, gh.SETS[set_name], rt, ops[1]))
        calls.append(lambda ops=ops: oz.check(oz.oz_dgemm_prepared(m, n, k, -1.0, ops[0], ops[1], 1.0, C, m, gh.SETS[set_name], rt)))
    assert _ratio(*calls) < 1.6
    gh.sync_status()


@pytest.mark.parametrize("set_name,sub", ROUTES)
@pytest.mark.parametrize("beta", [0.0, 1.0])
def test_odd_leading_dimension_of_the_residues(set_name, sub, beta):
    """Residues element by element, against the words that the next even leading dimension allows."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    m, n = 3001, 2999
    sA, sB = torch.zeros(m, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    C = _normal(m, n, 1)
    calls = []
    for ldr in (3001, 3008):
        R = _residues(set_name, n, ldr, None, 2)
        calls.append(lambda R=R, ldr=ldr: oz.check(oz.oz_reconstruct(m, n, R, ldr, n * ldr, sA, sB, gh.SETS[set_name], -1.0, beta, C, m)))
    assert _ratio(*calls) < 1.8


def test_wide_columns_of_a_small_operand():
    """Columns whose exponents spread, below the size from which a guess of their largest exponent pays."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    n, k, rt, S = 2647, 1700, gh.route("int8n"), gh.SETS["A"]
    block = torch.empty(oz.oz_operand_bytes(1, n, k, S, rt), dtype=torch.uint8, device="cuda")
    calls = []
    for sigma in (2.0, 0.0):
        X = _normal(k, n, 1) * torch.exp(sigma * _normal(k, n, 2))
        calls.append(lambda X=X: oz.check(oz.oz_prepare_operand(1, n, k, X, k, S, rt, block)))
    assert _ratio(*calls) < 1.05


def test_rows_of_zeros():
    """Rows of A without a normal number are read again for subnormals."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    m, k, rt, S = 6000, 12000, gh.route("int8n"), gh.SETS["A"]
    block = torch.empty(oz.oz_operand_bytes(0, m, k, S, rt), dtype=torch.uint8, device="cuda")
    X, Z = _normal(m, k, 1), _normal(m, k, 1)
    Z[:, ::10] = 0.0
    assert _ratio(*(lambda Y=Y: oz.check(oz.oz_prepare_operand(0, m, k, Y, m, S, rt, block)) for Y in (Z, X))) < 1.38


@pytest.mark.parametrize("set_name", ["S", "E"])
def test_reconstruction_on_the_tensor_pipe(set_name):
    """OZ_RECON_TENSOR against the default form: its integer tail may cost as much again as the whole call, its loads no more than that form's."""
    import torch

    import paper_2609_09095_b200 as oz
    import tests.gpu_helpers as gh
    m, n, k, S = 6000, 6000, 128, gh.SETS[set_name]
    A, B, C = _normal(m, k, 1), _normal(k, n, 2), torch.empty((n, m), dtype=torch.float64, device="cuda")
    gh.ensure_workspace(oz.oz_workspace_bytes(m, n, k, S, gh.route("fp8")))
    assert _ratio(*(lambda r=r: oz.check(oz.oz_dgemm_ex(m, n, k, 1.0, A, m, B, k, 0.0, C, m, S, gh.route("fp8", recon=r)))
                    for r in ("tensor", None))) < 2.2
