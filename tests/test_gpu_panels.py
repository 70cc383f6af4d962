"""The min-plus kernel at the edges of its panels, tiles and task words (run on a
GB300: pytest -m gpu).  With every output resolved exactly, its tables equal those
of the reference kernel, which the other tests hold to the oracle."""
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


# 15 column blocks of 64 make a panel with 7 or 8 multipliers, 16 with fewer: one block, a panel less one
# value, exactly, plus one, two panels and a remainder; s = 3 (one layer), s = 18 and 19 (128 tasks of 8
# multipliers and one more layer: two splits), s = 50 (four splits), s = 79 to 114 (one stage
# buffer of the skip test with 8 multipliers above s = 79).
@pytest.mark.parametrize("mode", ["DEFAULT", "RESIDENT_COSTS", "STREAMED_COSTS"])
@pytest.mark.parametrize("d,s,G", [(128, 3, 1), (959, 16, 8), (960, 16, 8), (961, 16, 7), (1024, 9, 5), (1025, 18, 6),
                                   (2000, 3, 8), (2113, 18, 8), (2113, 19, 8), (1984, 50, 8), (1100, 82, 8),
                                   (4097, 32, 3), (1100, 79, 8), (1100, 80, 8), (1100, 114, 8), (1100, 114, 7)])
def test_panel_edges_match_reference_kernel(E, mode, d, s, G):
    x = workloads.student_t(d, d + s, scale=1.0)
    lams = [0.0, 1e-4, 1e-3, 0.01, 0.05, 0.2, 1.0, 10.0][-G:]
    flags = getattr(E, mode, 0) | E.EXACT_TABLES
    wsr, ws = E.workspace(d, s), E.workspace(d, s, flags=flags)
    Qr, mr, metr = E.ecasq_dp_pass(x, s, lams, flags=E.DP_REFERENCE, ws=wsr)
    Q, m, met = E.ecasq_dp_pass(x, s, lams, flags=flags, ws=ws)
    st = E.native.ws_status(ws)
    assert st["timeout"] == 0 and st["bound_viol"] == 0
    assert m == mr
    np.testing.assert_array_equal(Q.cpu().numpy(), Qr.cpu().numpy())
    np.testing.assert_array_equal(met, metr)
    for g in range(G):
        for a, b in zip(E.ecasq_dp_tables(ws, g, s, d), E.ecasq_dp_tables(wsr, g, s, d)):
            np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())


def _far_tiles(fetched, nblocks, G, sms):
    """Of the cost tiles that a pass with a table copied in, the far phases'; and the most segments they can be in when four
    CTAs share a panel's."""
    pairs = (G + 1) // 2
    groups = lambda n: sum(b // 4 + 1 for b in range(n))  # tile groups of a panel's triangle
    T = max(n for n in range(1, 17) if groups(n) * pairs <= sms)
    panels = [min(T, nblocks - b) for b in range(0, nblocks, T)]
    return fetched - pairs * sum(n * (n + 1) // 2 for n in panels), sum(4 + n - 1 for n in panels[1:])


# A column block's far tiles reach the outputs in segments, a segment of more than 255 tiles in parts.  At most 16 tasks a
# tile make one entry of the far list; then far tiles beyond three a segment mean that segments had several parts.
@pytest.mark.parametrize("mode", ["DEFAULT", "RESIDENT_COSTS", "STREAMED_COSTS"])
@pytest.mark.parametrize("d,s,G,ties", [(2100, 4, 8, False), (4097, 4, 8, True), (4097, 10, 2, False), (6001, 10, 2, True),
                                        (3000, 16, 8, True), (2113, 19, 8, False)])
def test_segments_of_several_parts_match_reference_kernel(E, mode, d, s, G, ties):
    x = workloads.student_t(d, d + s, scale=1.0)
    if ties:  # evenly spaced values: wide bands, many tiles in a run and runs across parts
        x = (np.arange(d) % (d - 7)).astype(np.float32)
    lams = [0.0, 1e-4, 1e-3, 0.01, 0.05, 0.2, 1.0, 10.0][-G:]
    flags = getattr(E, mode, 0) | E.EXACT_TABLES
    wsr, ws, wsp = E.workspace(d, s), E.workspace(d, s, flags=flags), E.workspace(d, s, flags=flags)
    Qr, mr, metr = E.ecasq_dp_pass(x, s, lams, flags=E.DP_REFERENCE, ws=wsr)
    E.ecasq_dp_pass(x, s, lams, flags=flags, ws=ws)
    Q, m, met = E.ecasq_dp_pass(x, s, lams, flags=flags | E.TEST_SHORT_PARTS, ws=wsp)
    st, whole = E.native.ws_status(wsp), E.native.ws_status(ws)
    assert st["timeout"] == 0 and st["bound_viol"] == 0
    assert m == mr
    np.testing.assert_array_equal(Q.cpu().numpy(), Qr.cpu().numpy())
    np.testing.assert_array_equal(met, metr)
    for g in range(G):
        for a, b in zip(E.ecasq_dp_tables(wsp, g, s, d), E.ecasq_dp_tables(wsr, g, s, d)):
            np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
    assert st["members"] == whole["members"]  # the bands too
    if mode == "RESIDENT_COSTS" and (s - 2) * G <= 16:
        import torch
        far, segments = _far_tiles(st["tiles_fetched"], (st["p"] + 63) // 64, G,
                                   torch.cuda.get_device_properties(0).multi_processor_count)
        assert far > 3 * segments


# ||X||^2 beyond what fp32 costs hold: 1e38 (its multiples overflow), 1e63, 1e-31, 1e-57 (its gaps' squares vanish); 2^60 and 2^-60 are
# about the ends of the range that is taken as it is.
@pytest.mark.parametrize("mode", ["DEFAULT", "RESIDENT_COSTS", "STREAMED_COSTS"])
@pytest.mark.parametrize("scale", [1e17, 1e30, 1e-17, 1e-30, 2.0 ** 24, 2.0 ** 26, 2.0 ** -34, 2.0 ** -36, None])
def test_magnitudes_beyond_fp32_match_reference_kernel(E, mode, scale):
    d, s = 1500, 9
    x = (workloads.normal(d, 4).astype(np.float64) * (scale or 1.0)).astype(np.float32)
    x[::7] = x[0]
    if scale is None:  # a spread that no factor brings into fp32
        x[1], x[2] = 3e38, -3e38
    lams = [0.0, 1e-8, 1e-3, 0.1, 1.0, 1e3]
    flags = getattr(E, mode, 0)
    wsr, ws = E.workspace(d, s), E.workspace(d, s, flags=flags)
    Qr, mr, metr = E.ecasq_dp_pass(x, s, lams, flags=E.DP_REFERENCE, ws=wsr)
    Q, m, met = E.ecasq_dp_pass(x, s, lams, flags=flags | E.EXACT_TABLES, ws=ws)
    assert E.native.ws_status(ws)["bound_viol"] == 0
    assert m == mr
    np.testing.assert_array_equal(Q.cpu().numpy(), Qr.cpu().numpy())
    np.testing.assert_array_equal(met, metr)
    tables = [[t.cpu().numpy() for t in E.ecasq_dp_tables(wsr, g, s, d)] for g in range(len(lams))]
    for g in range(len(lams)):
        for a, b in zip(E.ecasq_dp_tables(ws, g, s, d), tables[g]):
            np.testing.assert_array_equal(a.cpu().numpy(), b)
    E.ecasq_dp_pass(x, s, lams, flags=flags, ws=ws)  # what is not resolved: the fp32 values, in x's own scale
    for g in range(len(lams)):
        dp, bp = (t.cpu().numpy() for t in E.ecasq_dp_tables(ws, g, s, d))
        np.testing.assert_allclose(dp[bp == -2], tables[g][0][bp == -2], rtol=1e-5)
        assert (bp == -2).any() or scale is None
    got, want = (E.ecasq_solve(x, s, budget_bits=1.7, refine_max_rounds=3, flags=f) for f in (flags, E.DP_REFERENCE))
    np.testing.assert_array_equal(got[0].cpu().numpy(), want[0].cpu().numpy())
    assert [got[1][k] for k in ("lambda", "mse", "h_exact")] == [want[1][k] for k in ("lambda", "mse", "h_exact")]
