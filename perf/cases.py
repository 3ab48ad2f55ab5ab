"""The work that programs have this library do, as cases that can be timed.

Every case is one call (or the pair of calls that a program makes per step) through the public entry
points of `paper_2609_09095_b200`: C = A B or C <- C - A B in emulated FP64 on device buffers, with the
operands of one side prepared once, or on pinned host buffers.  Matrices are column-major, held as
contiguous (columns, rows) tensors.

Fields of a case
  kind   "gemm" (oz_dgemm_ex), "prepared" (operator deconstructed once, oz_prepare_operand of the block and
         oz_dgemm_prepared per step), "host" (oz_dgemm_host on pinned buffers)
  m n k  shape;  pad: extra rows of the leading dimensions (a submatrix of a larger one)
  set    modulus set S, E or A;  sub: substrate of the residue products (fp8, int8 digits, int8n native)
  quant  RN or TZ;  rule: scale rule CS, MAXEXP or ACCURATE;  update: C <- C - A B instead of C = A B
  fallback  rows that fail the exponent-span check are re-issued in FP64 (OZ_FALLBACK_FP64)
  dist   entries: "uniform" U(-1,1), "normal" N(0,1), "lognormal:s" (U(0,1)-1/2) exp(s N(0,1)),
         "mixed" N(0,1) with three rows in a hundred of A lognormal:3 (badly scaled equations)
"""
import math

import torch

import paper_2609_09095_b200 as oz

SETS = {"S": oz.OZ_SET_S, "E": oz.OZ_SET_E, "A": oz.OZ_SET_A}
SUBS = {"fp8": oz.OZ_SUB_FP8, "int8": oz.OZ_SUB_INT8, "int8n": oz.OZ_SUB_INT8_NATIVE}
QUANTS = {"RN": oz.OZ_QUANT_RN, "TZ": oz.OZ_QUANT_TZ}
RULES = {"CS": oz.OZ_SCALE_CS, "MAXEXP": oz.OZ_SCALE_MAXEXP, "ACCURATE": oz.OZ_SCALE_ACCURATE}

BASE = {"kind": "gemm", "pad": 0, "set": "S", "sub": "fp8", "quant": "RN", "rule": "CS", "update": False,
        "fallback": False, "dist": "uniform"}


def _case(m, n, k, **fields):
    return {**BASE, "m": m, "n": n, "k": k, **fields}


def listed():
    return [
        # one small dense product, where latency and launches count (a block of a sparse or batched solver)
        {"name": "tiny_256", **_case(256, 256, 256)},
        # an ordinary odd-sized product
        {"name": "odd_1009", **_case(1009, 983, 1021)},
        # the square product of dense linear algebra, moderate exponent spread
        {"name": "square_4096", **_case(4096, 4096, 4096, dist="lognormal:0.5")},
        # HPL trailing update at the start of a factorisation (panel width 1024), the headline workload
        {"name": "hpl_update_16384", **_case(16384, 16384, 1024, update=True)},
        # a later trailing update of the same factorisation: a submatrix, hybrid set E
        {"name": "hpl_late_E", **_case(6912, 6912, 1024, set="E", update=True, pad=9472)},
        # the fastest route a program can choose: native INT8 residues of the all-byte set
        {"name": "native_int8_6144", **_case(6144, 6144, 3072, set="A", sub="int8n", dist="normal")},
        # tall-skinny block-Krylov product on INT8 digits
        {"name": "tall_int8", **_case(131072, 128, 4096, sub="int8", dist="normal")},
        # large ragged product with a wide exponent spread
        {"name": "ragged_10007", **_case(10007, 9973, 5003, dist="lognormal:2.0")},
        # block iterative solver: the operator's planes are kept, each step prepares and multiplies a block
        {"name": "krylov_prepared", **_case(10240, 64, 10240, kind="prepared", dist="normal")},
        # accurate mode: shifts from the extra bound product
        {"name": "accurate_2048", **_case(2048, 2048, 2048, rule="ACCURATE", dist="lognormal:0.5")},
        # badly scaled rows re-issued in FP64
        {"name": "fallback_2003", **_case(2003, 1999, 1501, fallback=True, dist="mixed")},
        # a trailing update on matrices that live in host memory
        {"name": "host_4096", **_case(4096, 4096, 1024, kind="host", update=True)},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _passes(case):
    r = {"S": 12, "E": 13, "A": 15}[case["set"]]
    return r if case["sub"] == "int8n" else 3 * r


def draw(rng):
    dist = rng.choice(["uniform", "normal", "lognormal:0.5", "lognormal:1.0"])
    route = dict(rng.choice([{"set": "S", "sub": "fp8"}, {"set": "S", "sub": "fp8"}, {"set": "S", "sub": "int8"},
                             {"set": "E", "sub": "fp8"}, {"set": "E", "sub": "int8"}, {"set": "A", "sub": "fp8"},
                             {"set": "A", "sub": "int8n"}]))
    route.update(quant=rng.choice(["RN", "RN", "TZ"]), rule=rng.choice(["CS", "CS", "CS", "MAXEXP"]), dist=dist)
    family = rng.choice(["small", "small", "square", "square", "update", "tall", "prepared", "accurate", "fallback", "host"])
    while True:
        if family == "small":
            c = _case(_log(rng, 64, 1500), _log(rng, 64, 1500), _log(rng, 64, 1500), update=rng.random() < 0.5, **route)
        elif family == "square":
            c = _case(_log(rng, 1000, 10000), _log(rng, 1000, 10000), _log(rng, 1000, 10000), **route)
        elif family == "update":
            c = _case(_log(rng, 1000, 16384), _log(rng, 1000, 16384), rng.choice([128, 256, 384, 512, 1024]), update=True,
                      pad=rng.choice([0, 1, 64, 1000]), **route)
        elif family == "tall":
            c = _case(_log(rng, 10000, 131072), _log(rng, 8, 256), _log(rng, 500, 4096), **route)
        elif family == "prepared":
            c = _case(_log(rng, 1000, 12000), _log(rng, 8, 512), _log(rng, 1000, 12000), kind="prepared", **route)
        elif family == "accurate":
            c = _case(_log(rng, 200, 5000), _log(rng, 200, 5000), _log(rng, 200, 5000), **{**route, "rule": "ACCURATE"})
        elif family == "fallback":
            c = _case(_log(rng, 300, 3000), _log(rng, 300, 3000), _log(rng, 300, 3000), fallback=True,
                      **{**route, "rule": "CS", "dist": "mixed"})
        else:
            c = _case(_log(rng, 300, 5000), _log(rng, 300, 5000), _log(rng, 200, 2000), kind="host",
                      update=rng.random() < 0.5, **route)
        if work(c)["flops"] <= 3e13 and c["m"] * c["k"] <= 131072 * 4096:
            return c


def _route(case):
    return (SUBS[case["sub"]] | QUANTS[case["quant"]] | RULES[case["rule"]] |
            (oz.OZ_FALLBACK_FP64 if case["fallback"] else 0))


def _entries(gen, rows, cols, dist, pad=0):
    """rows x cols, column-major with leading dimension rows + pad: a contiguous (cols, rows + pad) tensor."""
    shape = (cols, rows + pad)
    new = dict(dtype=torch.float64, device="cuda", generator=gen)
    if dist == "uniform":
        return torch.rand(shape, **new).mul_(2.0).sub_(1.0)
    x = torch.randn(shape, **new)
    if dist.startswith("lognormal:"):
        return x.mul_(float(dist.split(":")[1])).exp_().mul_(torch.rand(shape, **new).sub_(0.5))
    if dist == "mixed":
        bad = torch.rand(rows + pad, **new) < 0.03
        x[:, bad] = _entries(gen, int(bad.sum()), cols, "lognormal:3")
    return x


# One workspace for the whole program, as large as its largest call needs.
_workspace = None


def _need_workspace(nbytes):
    global _workspace
    if _workspace is None or _workspace.numel() < nbytes:
        oz.oz_set_workspace(None)
        _workspace = None
        _workspace = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        oz.check(oz.oz_set_workspace(_workspace), "oz_set_workspace")


def prepare(case, seed):
    m, n, k, pad = case["m"], case["n"], case["k"], case["pad"]
    modset, route = SETS[case["set"]], _route(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    A = _entries(gen, m, k, case["dist"], pad)
    B = _entries(gen, k, n, "normal" if case["dist"] == "mixed" else case["dist"], pad)
    C = _entries(gen, m, n, "uniform", pad)
    s = {"kind": case["kind"], "m": m, "n": n, "k": k, "ld": pad, "set": modset, "route": route,
         "alpha": -1.0 if case["update"] else 1.0, "beta": 1.0 if case["update"] else 0.0}
    if case["kind"] == "prepared":
        _need_workspace(oz.oz_product_workspace_bytes(m, n, modset))
        s["opA"] = torch.empty(oz.oz_operand_bytes(0, m, k, modset, route), dtype=torch.uint8, device="cuda")
        s["opB"] = torch.empty(oz.oz_operand_bytes(1, n, k, modset, route), dtype=torch.uint8, device="cuda")
        oz.check(oz.oz_prepare_operand(0, m, k, A, m + pad, modset, route, s["opA"]), "oz_prepare_operand")
        s.update(B=B, C=C)
    elif case["kind"] == "host":
        _need_workspace(oz.oz_workspace_bytes(m, n, k, modset, route) + 8 * (m * k + k * n + m * n) + 4096)
        s.update({name: torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
                  for name, x in (("A", A), ("B", B), ("C", C))})
    else:
        _need_workspace(oz.oz_workspace_bytes(m, n, k, modset, route))
        s.update(A=A, B=B, C=C)
    return s


def run(s):
    m, n, k, C = s["m"], s["n"], s["k"], s["C"]
    lda = ldc = m + s["ld"]
    ldb = k + s["ld"]
    if s["kind"] == "prepared":
        oz.check(oz.oz_prepare_operand(1, n, k, s["B"], ldb, s["set"], s["route"], s["opB"]), "oz_prepare_operand")
        oz.check(oz.oz_dgemm_prepared(m, n, k, s["alpha"], s["opA"], s["opB"], s["beta"], C, ldc, s["set"], s["route"]),
                 "oz_dgemm_prepared")
    elif s["kind"] == "host":
        oz.check(oz.oz_dgemm_host(m, n, k, s["alpha"], s["A"], lda, s["B"], ldb, s["beta"], C, ldc, s["set"], s["route"]),
                 "oz_dgemm_host")
        torch.cuda.current_stream().synchronize()      # the program goes on to read C on the host
    else:
        oz.check(oz.oz_dgemm_ex(m, n, k, s["alpha"], s["A"], lda, s["B"], ldb, s["beta"], C, ldc, s["set"], s["route"]),
                 "oz_dgemm_ex")
    return C


def work(case):
    """Operands and C moved once (planes of the kept operator for "prepared"); the plane products of the
    method (3 r, or r on native residues; one more in accurate mode), 2 m n k operations each."""
    m, n, k = case["m"], case["n"], case["k"]
    stored = {"S": 30, "E": 33, "A": 44}[case["set"]] if case["sub"] != "int8n" else 15
    a_bytes = (stored if case["kind"] == "prepared" else 8) * m * k
    passes = _passes(case) + (1 if case["rule"] == "ACCURATE" else 0)
    return {"bytes": a_bytes + 8 * k * n + (16 if case["update"] else 8) * m * n, "flops": passes * 2 * m * n * k}


def tolerance(case):
    """The shifts fix the integer product c' and C is its correctly rounded value (then one FP64 addition in
    an update), and the re-issued rows are a compensated sum in a fixed order: one result, bit for bit."""
    return "exact"
