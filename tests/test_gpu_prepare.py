"""The preparation's exact sums (run on a GB300: pytest -m gpu): lengths around a thread's, a
block's and several blocks' keys; ranges that fill the integer window, just miss it, or hold
denormals.  The prefixes are the exact sums rounded once to double-doubles where the window holds."""
from fractions import Fraction

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


def _prefixes(x, scale):
    """Exact prefix sums of the integers x (units 2^-scale) as double-doubles: nearest, then nearest rest."""
    hi, lo, run = [0.0], [0.0], 0
    for v in x:
        run += v
        h = run / (1 << scale)
        hi.append(h)
        lo.append((run - int(Fraction(h) * (1 << scale))) / (1 << scale))
    return np.array(hi), np.array(lo)


@pytest.mark.parametrize("d", [1, 2, 15, 16, 17, 255, 4095, 4096, 4097, 8193, 20001])
@pytest.mark.parametrize("kind", ["normal", "octaves80", "octaves200", "denormal", "repeated", "zeros"])
def test_prefix_sums_are_exact_sums_rounded_once(E, d, kind):
    rng = np.random.default_rng(d)
    x = rng.standard_normal(d).astype(np.float32)
    if kind.startswith("octaves"):
        x = np.ldexp(x, rng.integers(-int(kind[7:]) // 2, int(kind[7:]) // 2 - 40, d)).astype(np.float32)
    elif kind == "denormal":
        x = (rng.integers(-1000, 1000, d) * 1.4e-45).astype(np.float32)
    elif kind == "repeated":
        x = rng.integers(-3, 4, d).astype(np.float32)
    elif kind == "zeros":
        x[:] = 0.0
    o = E.ecasq_prepare(x)
    v, n = np.unique(x + np.float32(0.0), return_counts=True)
    p = v.size
    assert o["p"] == p
    np.testing.assert_array_equal(o["v"].cpu().numpy()[:p], v)
    np.testing.assert_array_equal(o["w"].cpu().numpy()[:p], n)
    np.testing.assert_array_equal(o["N"].cpu().numpy()[:p + 1], np.concatenate([[0], np.cumsum(n)]))
    k = [int(Fraction(float(a)) * (1 << 149)) for a in v]
    for name, terms, scale in (("S", [a * int(b) for a, b in zip(k, n)], 149), ("S2", [a * a * int(b) for a, b in zip(k, n)], 298)):
        hi, lo = o[name + "_hi"].cpu().numpy(), o[name + "_lo"].cpu().numpy()
        ehi, elo = _prefixes(terms, scale)
        if kind == "octaves200":  # beyond the window: double-double sums of d terms
            np.testing.assert_allclose(hi, ehi, rtol=2.0 ** -50 if name == "S2" else 0, atol=2.0 ** -50 * np.abs(ehi).max())
        else:
            np.testing.assert_array_equal(hi, ehi, err_msg=name)
            np.testing.assert_array_equal(lo, elo, err_msg=name)
