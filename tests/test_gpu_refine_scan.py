"""The refinement's scans (run on a GB300: pytest -m gpu).  The full scan of inputs of at most 512 unique
values an SM: blocks of 32 and 64 candidates and their edges, neighbours with one or no candidate between
them, data of every kind below, multipliers that leave costs or entropies alone.  The screened scan
of larger ones: blocks of 64, 128 and 256, data whose offset, outliers, magnitude or repetition make the
screening's error bound wide, the same multipliers.  Codebooks, rounds and objectives equal the oracle's,
from a start far from the optimum."""
import numpy as np
import pytest

from paper_2608_18147_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    import paper_2608_18147_gb300 as E
    E.lib()
    return E


@pytest.mark.parametrize("kind", ["normal", "offset", "outliers", "tiny", "huge", "repeated", "integers"])
@pytest.mark.parametrize("d,m", [(5, 5), (40, 16), (258, 3), (259, 4), (1025, 9), (4099, 16), (3000, 40), (90001, 9)])
def test_refinement_equals_the_oracle(E, oracle_mod, d, m, kind):
    rng = np.random.default_rng(d + m)
    x = workloads.normal(d, d)
    if kind == "offset":
        x = (x + np.float32(1e4)).astype(np.float32)
    elif kind == "outliers":
        x[:3] = np.array([-3e9, 2e12, 5e12], np.float32)
    elif kind == "tiny":
        x = (x * np.float32(1e-30)).astype(np.float32)
    elif kind == "huge":
        x = (x * np.float32(1e17)).astype(np.float32)
    elif kind == "repeated":
        x = np.round(x * 50) / np.float32(50)
    elif kind == "integers":
        x = np.cumsum(rng.integers(1, 40, d)).astype(np.float32)
    H = oracle_mod.Hist(x)
    if d < 40000:
        H.cache()
    v = H.arrays()["v"]
    p = v.size
    m = min(m, p)
    a0 = np.unique(np.concatenate([[0, p - 1], np.linspace(0, p - 1, m).astype(int)]))
    if a0.size > 4:
        a0[2] = a0[1] + 1  # neighbours next to one another
    a0 = np.unique(a0).astype(np.int32)
    for lam in (0.0, 1e-4, 0.05, 30.0) if d < 40000 else (1e-3,):
        o = H.refine(a0, lam * H.norm2, budget=np.inf, guard=False, max_rounds=5, tol=0.0)
        Q, res = E.ecasq_refine(x, v[a0], lam, budget_bits=-1.0, max_rounds=5, rel_tol=0.0)
        np.testing.assert_array_equal(Q.cpu().numpy(), v[o["Q_idx"]], err_msg=str(lam))
        assert res["refine_rounds"] == o["rounds"]
        if len(o["J"]):
            np.testing.assert_allclose(res["objective"], o["J"][-1], rtol=1e-9,
                                       atol=2.0 ** -90 * H.norm2)  # double-double differences of ||X||^2


def _large(kind):
    """More than 80 000 distinct values."""
    rng, x = np.random.default_rng(4), workloads.normal(90001, 90001)
    if kind == "cluster":      # far from zero, a few last places apart
        x = (1e4 + rng.uniform(0, 2000, x.size)).astype(np.float32)
    elif kind == "integers":   # about 2^23
        x = (2.0 ** 23 - 1e6 + np.cumsum(rng.integers(1, 40, x.size))).astype(np.float32)
    elif kind == "outliers":
        x[:3] = np.array([-3e9, 2e12, 5e12], np.float32)
    elif kind == "tiny":
        x = x * np.float32(1e-30)
    elif kind == "huge":
        x = x * np.float32(1e17)
    elif kind == "repeated":
        v = np.unique(x)[:85000]
        x = np.concatenate([v, rng.choice(v[:2000], 40000)])
    return x


# (9 values: blocks of 64 candidates; 70: 128; 140: 256; one size smaller for the repeated ones)
@pytest.mark.parametrize("kind,m", [(k, m) for k in ("normal", "cluster", "integers", "outliers", "tiny", "huge", "repeated")
                                    for m in (9, 140)] + [("cluster", 70), ("repeated", 70)])
def test_screened_refinement_equals_the_oracle(E, oracle_mod, kind, m):
    import torch
    x = _large(kind)
    H = oracle_mod.Hist(x)
    v = H.arrays()["v"]
    p = v.size
    assert p > 512 * torch.cuda.get_device_properties(0).multi_processor_count  # else the full scan runs
    a0 = np.unique(np.concatenate([[0, p - 1], np.linspace(0, p - 1, m).astype(int)])).astype(np.int32)
    a0[2] = a0[1] + 1  # neighbours next to one another
    for lam in (0.0, 1e-3, 30.0):
        o = H.refine(a0, lam * H.norm2, budget=np.inf, guard=False, max_rounds=3, tol=0.0)
        Q, res = E.ecasq_refine(x, v[a0], lam, budget_bits=-1.0, max_rounds=3, rel_tol=0.0)
        np.testing.assert_array_equal(Q.cpu().numpy(), v[o["Q_idx"]], err_msg=str(lam))
        assert res["refine_rounds"] == o["rounds"]
        np.testing.assert_allclose(res["objective"], o["J"][-1], rtol=1e-9,
                                   atol=2.0 ** -90 * H.norm2)  # double-double differences of ||X||^2
