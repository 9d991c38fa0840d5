"""Binning of large batches, eight lanes per (spectrum, bin): bins of three to four hundred entries,
overlapping and out of order, and batch sizes that leave the last block part full, with and without
uncertainties.

Bar: sums of at most about 400 positive FP64 terms in another order, and a square root:
relative 1e-12."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1912_07759_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_bin", [(683, 12), (2731, 3), (9001, 1)])
def test_large_batches_match_the_oracle(B, n_bin):
    import torch
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(1, 1, 4, 4, 3000, with_cia=False)
    tables = T.XsecTables(ctx, tb)
    rng = np.random.default_rng(n_bin)
    centre = rng.uniform(0.5, 5.0, n_bin)
    width = centre * np.geomspace(0.004, 0.6, n_bin)
    bins = T.Bins(ctx, tables, centre, width)
    i0, i1 = bins.native_range
    flux = rng.uniform(0.01, 0.02, (B, i1 - i0))
    sig = rng.uniform(1e-5, 1e-4, (B, i1 - i0))
    f, s = T.bin_spectra(ctx, bins, torch.tensor(flux, device="cuda"),
                         torch.tensor(sig, device="cuda"), base=i0)
    few = [0, 1, B // 2, B - 1]
    native = np.zeros((2, len(few), tb.n_wn))
    native[0, :, i0:i1], native[1, :, i0:i1] = flux[few], sig[few]
    rf, rs = O.bin_with_uncertainty(tb.wn_grid, centre, width, native[0], native[1])
    assert np.allclose(f.cpu().numpy()[few], rf, rtol=1e-12, atol=0)
    assert np.allclose(s.cpu().numpy()[few], rs, rtol=1e-12, atol=0)
    # every spectrum as in a batch too small for this form
    for b in range(0, B, 997):
        f1, s1 = T.bin_spectra(ctx, bins, torch.tensor(flux[b:b + 1], device="cuda"),
                               torch.tensor(sig[b:b + 1], device="cuda"), base=i0)
        assert np.allclose(f1.cpu().numpy()[0], f[b].cpu().numpy(), rtol=1e-12, atol=0)
        assert np.allclose(s1.cpu().numpy()[0], s[b].cpu().numpy(), rtol=1e-12, atol=0)
