"""The short-codebook encodes where they can go wrong (run on a GB300: pytest -m gpu):
lengths around a group of four and a block's step, misaligned inputs, pairs of
codebooks of different sizes and ranges, and what they refuse.  Bit-exact against the
oracle."""
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


def _case(d, mm, mp, seed, narrow):
    """Codebooks over [-4, 4] (the second over [-2, 2] when narrow), entries of both among the inputs."""
    rng = np.random.default_rng(seed)
    book = lambda m, r: np.sort(np.concatenate([[-r, r][:m], rng.uniform(-r, r, max(m - 2, 0))])).astype(np.float32)
    Qm, Qp = book(mm, 4.0), book(mp, 2.0 if narrow else 4.0)
    lim = 0.0 if min(mm, mp) == 1 else (1.99 if narrow else 3.99)
    x = rng.uniform(-lim, lim, d).astype(np.float32)
    if min(mm, mp) > 1:
        pick = np.concatenate([Qm[np.abs(Qm) <= lim], Qp[np.abs(Qp) <= lim], [0.0, 1e-40]]).astype(np.float32)
        x[::3] = rng.choice(pick, x[::3].size)
    else:
        Qm, Qp = Qm[:mm] if mm > 1 else np.zeros(1, np.float32), Qp[:mp] if mp > 1 else np.zeros(1, np.float32)
    return x, Qm, Qp


@pytest.mark.parametrize("d,offset", [(1, 0), (3, 0), (5, 0), (2047, 0), (2049, 1), (4096, 0), (4103, 3), (3000001, 0)])
@pytest.mark.parametrize("mm,mp,beta,narrow", [(1, 2, 0.5, False), (16, 16, 0.563, False), (3, 9, 0.0, True),
                                               (16, 5, 1.0, True), (7, 16, 2.0 ** -24, True), (16, 17, 0.3, False)])
def test_pairs_of_codebooks_bit_exact(E, oracle_mod, d, offset, mm, mp, beta, narrow):
    import torch
    x, Qm, Qp = _case(d, mm, mp, 7 * d + mm, narrow)
    xt = torch.zeros(d + offset, dtype=torch.float32, device="cuda")
    xt[offset:] = torch.as_tensor(x).cuda()
    for with_sel in (True, False):
        idx, sel, counts, rate = E.ecasq_quantize_timeshare(xt[offset:], Qm, Qp, beta, 11, 12, with_sel=with_sel)
        oi, os_, oc, orate = oracle_mod.quantize_timeshare(x, Qm, Qp, beta, 11, 12)
        np.testing.assert_array_equal(idx.cpu().numpy(), oi)
        if with_sel:
            np.testing.assert_array_equal(sel.cpu().numpy(), os_)
        np.testing.assert_array_equal(counts.cpu().numpy().astype(np.uint32), oc)
        assert rate == pytest.approx(orate, rel=1e-12, abs=1e-15)


@pytest.mark.parametrize("m", [4, 16, 20, 40])
def test_refusals_and_small_workspace(E, oracle_mod, m):
    """A codebook out of order and an entry outside it are refused whatever the size; a workspace that
    holds the status record alone gives the same counts."""
    import torch
    Q = np.linspace(-1, 1, m).astype(np.float32)
    x = np.random.default_rng(m).uniform(-1, 1, 9001).astype(np.float32)
    oi, oc, oh = oracle_mod.quantize(x, Q, 3)
    for nbytes in (128, 4096):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        idx, counts, h = E.ecasq_quantize(x, Q, 3, ws=ws)
        np.testing.assert_array_equal(idx.cpu().numpy(), oi)
        np.testing.assert_array_equal(counts.cpu().numpy().astype(np.uint32), oc)
        assert h == pytest.approx(oh, rel=1e-12)
        for bad in (Q[::-1].copy(), np.concatenate([Q[:-1], [Q[-2]]]).astype(np.float32),
                    np.where(np.arange(m) == 1, np.nan, Q).astype(np.float32)):
            with pytest.raises(E.EcasqError) as ei:
                E.ecasq_quantize(x, bad, 3, ws=ws)
            assert ei.value.code == E.native.EINVAL
            with pytest.raises(E.EcasqError) as ei:
                E.ecasq_quantize_timeshare(x, Q, bad, 0.5, 3, 4, ws=ws)
            assert ei.value.code == E.native.EINVAL
        for v, at in ((1.5, 0), (np.nan, 4500), (-np.inf, 9000)):
            y = x.copy()
            y[at] = v
            with pytest.raises(E.EcasqError) as ei:
                E.ecasq_quantize(y, Q, 3, ws=ws)
            assert ei.value.code == E.native.ERANGE


@pytest.mark.parametrize("m", [2, 16, 17])
@pytest.mark.parametrize("d", [7, 8, 4096, 9001])
@pytest.mark.parametrize("part", [0, 1])
def test_a_nan_codebook_of_one_value_is_out_of_range(E, d, m, part):
    """No entry lies within a codebook whose one value is NaN: refused whichever kernel meets the entry,
    and no matter for the part that no entry takes."""
    x = np.random.default_rng(d).uniform(-1, 1, d).astype(np.float32)
    Q, nan = np.linspace(-1, 1, m).astype(np.float32), np.array([np.nan], np.float32)
    Qm, Qp = (nan, Q) if part == 0 else (Q, nan)
    with pytest.raises(E.EcasqError) as ei:
        E.ecasq_quantize_timeshare(x, Qm, Qp, 0.5, 3, 4)
    assert ei.value.code == E.native.ERANGE
    idx, sel, counts, _ = E.ecasq_quantize_timeshare(x, Qm, Qp, 1.0 - part, 3, 4)
    other = E.ecasq_quantize(x, Q, 3)
    np.testing.assert_array_equal(idx.cpu().numpy(), other[0].cpu().numpy())
    np.testing.assert_array_equal(counts.cpu().numpy()[1:] if part == 0 else counts.cpu().numpy()[:-1],
                                  other[1].cpu().numpy())


@pytest.mark.parametrize("m", [1, 2, 4, 5, 9, 16, 17, 40])
def test_an_infinite_last_value_keeps_to_its_codebook(E, oracle_mod, m):
    """A codebook that ends in +inf and entries equal to it: the last index, and nothing written behind the counts."""
    import torch
    Q = np.concatenate([np.linspace(-1, 1, max(m - 1, 1)), [np.inf]])[-m:].astype(np.float32)
    rng = np.random.default_rng(m)
    for d in (6, 9001):
        x = (rng.uniform(-1, 1, d) if m > 2 else np.full(d, np.inf)).astype(np.float32)
        x[1::5] = np.inf
        oi, oc, _ = oracle_mod.quantize(x, Q, 3)
        for nbytes in (128, 4096):  # the counts in the caller's buffer, or behind the status record
            ws = torch.full((nbytes + 256,), 0x5A, dtype=torch.uint8, device="cuda")
            out = torch.full((64,), -7, dtype=torch.int32, device="cuda")
            idx, _, _ = E.ecasq_quantize(x, Q, 3, ws=ws[:nbytes], counts=out[:m])
            np.testing.assert_array_equal(idx.cpu().numpy(), oi)
            np.testing.assert_array_equal(out[:m].cpu().numpy(), oc.astype(np.int32))
            assert bool((out[m:] == -7).all()) and bool((ws[nbytes:] == 0x5A).all())
        for Qm, Qp in ((Q, Q), (Q, np.array([-1, 0.5, np.inf], np.float32))):
            if Qp[0] > x.min():
                continue
            idx, sel, counts, _ = E.ecasq_quantize_timeshare(x, Qm, Qp, 0.4, 3, 4)
            oi2, os2, oc2, _ = oracle_mod.quantize_timeshare(x, Qm, Qp, 0.4, 3, 4)
            np.testing.assert_array_equal(idx.cpu().numpy(), oi2)
            np.testing.assert_array_equal(sel.cpu().numpy(), os2)
            np.testing.assert_array_equal(counts.cpu().numpy().astype(np.uint32), oc2)
