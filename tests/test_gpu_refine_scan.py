"""The refinement's scans (run on a GB300: pytest -m gpu): the screened one of large inputs and the
full one of small ones, chunks of 256 candidates and their edges, neighbours with one or no candidate between them, data whose offset, outliers, magnitude or
repetition make the screening's error bound wide, and multipliers that leave costs or entropies
alone.  Codebooks, rounds and objectives equal the oracle's, from a start far from the optimum."""
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
