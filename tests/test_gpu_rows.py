"""The batched rows' pass where it can go wrong (run on a GB300: pytest -m gpu): rows around the
size whose costs fit shared memory and around units of 32 columns, up to the longest; codebook
sizes around a warp; ties; magnitudes and gaps at the ends of the fp32 range.  Every row equals the
single solve with the binary64 kernel."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    import paper_2608_18147_gb300 as E
    E.lib()
    return E


def _same(E, X, s, **kw):
    flags = kw.pop("flags", 0)
    Q, m, res = E.ecasq_solve_batched(X, s, flags=flags, **kw)
    Q, m = Q.cpu().numpy(), m.cpu().numpy()
    for r in range(X.shape[0]):
        Q1, r1 = E.ecasq_solve(X[r], s, flags=flags | E.DP_REFERENCE, **kw)
        assert m[r] == r1["m"], r
        np.testing.assert_array_equal(Q[r, :m[r]], Q1.cpu().numpy(), err_msg=f"row {r}")
        for key in ("status", "lambda", "mse", "h_surrogate", "h_exact", "p", "passes", "lambdas_evaluated"):
            assert res[r][key] == r1[key], (r, key)


@pytest.mark.parametrize("d,s", [(2, 2), (31, 3), (33, 8), (127, 8), (128, 16), (129, 8), (160, 2), (161, 33), (300, 8),
                                 (513, 5), (1023, 16), (1024, 8)])
def test_rows_equal_the_binary64_solve(E, d, s):
    rng = np.random.default_rng(d)
    X = rng.standard_normal((5, d)).astype(np.float32)
    X[1] = rng.standard_t(2, d).astype(np.float32)
    X[2] = np.round(X[2] * 40) / 40                          # repeated values, evenly spaced: ties
    X[3] = np.arange(d, dtype=np.float32) - d // 3           # every interval of one length ties
    X[4] = np.exp(3 * X[4])
    _same(E, X, s, budget_bits=1.5)
    if d in (33, 129, 300):
        _same(E, X, s, budget_bits=2.0, flags=E.EXACT_S)
        _same(E, X, s, lambda_=0.0)
        _same(E, X, s, lambda_=0.3)


@pytest.mark.parametrize("d", [60, 128, 200])
def test_rows_at_the_ends_of_the_fp32_range(E, d):
    """Magnitudes of 1e18 and 1e-18, values 1e-30 of the largest, gaps too small for fp32 costs
    (binary64 costs, rounded) and a multiplier beyond fp32."""
    rng = np.random.default_rng(9)
    X = rng.standard_normal((6, d)).astype(np.float32)
    X[0] *= np.float32(1e18)
    X[1] *= np.float32(1e-18)
    X[2, : d // 2] *= np.float32(1e-30)
    X[3, : d // 2] = (np.arange(d // 2) * 1.4e-45).astype(np.float32)
    X[4, 0], X[4, 1] = np.float32(3e38), np.float32(-3e38)
    X[5] = np.linspace(0, 1e-40, d).astype(np.float32)
    _same(E, X, 6, budget_bits=1.5)
    _same(E, X[:3], 6, lambda_=1e37)


def test_a_value_that_is_not_finite_refuses_every_group(E):
    """More rows than are searched together: a NaN in the last one leaves every row's results unwritten."""
    import torch
    rows, d, s = 300, 1024, 4
    X = torch.as_tensor(np.random.default_rng(5).standard_normal((rows, d)).astype(np.float32)).cuda()
    X[299, 17] = float("nan")
    ws = E.workspace(d, s, rows)
    Q = torch.full((rows, s), 7.0, device="cuda")
    m = torch.full((rows,), 7, dtype=torch.int32, device="cuda")
    prm, ptr = E.native.make_params(s, 1.5), E.native._ptr
    rc = E.lib().ecasq_solve_batched(ptr(X), rows, d, C.byref(prm), ptr(ws), ws.numel(), ptr(Q), ptr(m), None,
                                     E.native._stream())
    torch.cuda.synchronize()
    assert rc == E.native.ENONFINITE
    assert bool((Q == 7).all()) and bool((m == 7).all())
    X[299, 17] = 0.25
    Qg, mg, res = E.ecasq_solve_batched(X, s, budget_bits=1.5, ws=ws)
    Q1, r1 = E.ecasq_solve(X[299], s, budget_bits=1.5)
    assert mg[299] == r1["m"] and res[299]["mse"] == r1["mse"]
    np.testing.assert_array_equal(Qg[299, : r1["m"]].cpu().numpy(), Q1.cpu().numpy())


@pytest.mark.parametrize("rows,d,flags", [(5, 100, 0), (5, 300, 0), (260, 1024, 0), (5, 300, "TIME_KERNELS")])
def test_rows_check_their_certificate(E, rows, d, flags):
    """The status record tells how many candidates the call evaluated in binary64 (over all rows, in groups or one by
    one) and that no fp32 value left its certified error."""
    flags = getattr(E, flags) if flags else 0
    rng = np.random.default_rng(d)
    X = rng.standard_normal((rows, d)).astype(np.float32)
    X[3] = np.arange(d)                                      # ties: many members an output
    X[4] = 1 + rng.integers(0, 40, d) * 2.0 ** -23           # neighbours far from zero
    ws = E.workspace(d, 8, rows, flags=flags)
    ws.fill_(0xFF)
    _, _, res = E.ecasq_solve_batched(X, 8, budget_bits=2.0, flags=flags, ws=ws)
    st = E.native.ws_status(ws)
    assert st["bound_viol"] == 0 and st["timeout"] == 0
    assert st["rescored"] > rows
    if flags:
        assert st["rescored"] >= sum(r["rescored"] for r in res)


@pytest.mark.parametrize("d,s", [(1024, 5), (1024, 6), (612, 16), (614, 16), (400, 38), (1024, 33)])
def test_one_long_row_alone(E, d, s):
    """Around the line from which the single solve takes one row."""
    X = np.random.default_rng(s).standard_normal((1, d)).astype(np.float32)
    X[0, :3] = 0.5  # (two values fewer)
    _same(E, X, s, budget_bits=1.5)
    _same(E, X, s, lambda_=0.3)
    X[0, 1:3] = [0.25, 0.75]
    _same(E, X, s, budget_bits=1.5)


@pytest.mark.parametrize("kw", [dict(lambda_=0.3), dict(lambda_=1e30), dict(lambda_=0.3, refine_max_rounds=2)])
def test_rows_without_a_codebook(E, kw):
    """Exactly s values from fewer: status and sizes whichever path a row takes (1e30 is beyond fp32, refinement goes row
    by row), and m = 0."""
    import torch
    X = np.random.default_rng(2).standard_normal((3, 9)).astype(np.float32)
    X[1] = np.round(X[1])
    rows, d = X.shape
    ws = E.workspace(d, 17, rows)
    prm, ptr = E.native.make_params(17, flags=E.EXACT_S, **kw), E.native._ptr
    Q, m = torch.zeros((rows, 17), device="cuda"), torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    Xd, res = torch.as_tensor(X).cuda(), (E.native.Result * rows)()
    C.memset(res, 0x5A, C.sizeof(res))
    rc = E.lib().ecasq_solve_batched(ptr(Xd), rows, d, C.byref(prm), ptr(ws), ws.numel(), ptr(Q), ptr(m),
                                     res, E.native._stream())
    assert rc == E.native.EINFEASIBLE
    assert m.cpu().numpy().tolist() == [0] * rows
    for r in range(rows):
        got = res[r].as_dict()
        assert got["status"] == E.native.EINFEASIBLE and got["m"] == 0 and got["d"] == d and got["passes"] == 0
        if not kw.get("refine_max_rounds"):
            assert got["p"] == np.unique(X[r]).size


@pytest.mark.parametrize("d,s", [(9, 5), (31, 12), (64, 16), (107, 64), (128, 40), (129, 64), (300, 33)])
def test_rows_that_tie(E, d, s):
    """Evenly spaced values, repeated ones and few distinct gaps: outputs tie by the thousand, layers of a closure from one
    output to whole rows, traces that meet outputs they resolved before."""
    rng = np.random.default_rng(d + s)
    X = np.tile(np.arange(d, dtype=np.float32), (5, 1))
    X[1] = X[1] * np.float32(0.1) - np.float32(d / 3)
    X[2] = rng.integers(-d // 3, d // 3, d)
    X[3] = np.cumsum(rng.integers(1, 3, d))
    X[4, : d // 2] = 2 * X[4, : d // 2]
    _same(E, X, s, lambda_=0.0)
    _same(E, X, s, lambda_=1e-3)
    _same(E, X, s, budget_bits=min(2.0, 0.6 * np.log2(s)))
    enough = [x for x in X if np.unique(x).size >= s]
    _same(E, np.stack(enough), s, budget_bits=min(3.0, 0.8 * np.log2(s)), flags=E.EXACT_S)


@pytest.mark.parametrize("d,s", [(11, 64), (13, 32), (40, 33), (130, 64)])
@pytest.mark.parametrize("kw", [dict(lambda_=0.0), dict(lambda_=1e-6), dict(budget_bits=1.7)])
def test_rows_whose_least_cost_is_rounding(E, d, s, kw):
    # magnitudes from 1e-20 to 1e17: past the last codeword that matters, double-double costs are rounding (2^-100 of ||X||^2)
    # and tie or differ by it, where fp32's are exactly zero or ordered
    rng = np.random.default_rng(1000 * d + s)
    X = rng.standard_normal((24, d))
    X[:, : d // 3] *= 1e17
    X[:, d // 3 : d // 3 + 3] *= 1e-20
    X[1::2] = X[1::2, ::-1] + 0.0
    _same(E, X.astype(np.float32), s, **kw)
