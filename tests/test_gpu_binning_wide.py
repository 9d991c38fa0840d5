"""Binning of large batches of wide bins: a batch takes no longer than its halves, whose spectra and
bins are too few for the form that large batches of narrow bins take; and around the line between
the two forms (a longest bin of 1,280 entries) and with one wide bin among narrow ones, the binned
spectra are the oracle's (relative 1e-12: sums of positive FP64 terms in another order)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def bins_of(n_bin, entries, n_wn, lam=0.4):
    """n_bin neighbouring bins of `entries` wavenumbers each of the log-uniform 300-30,000 grid."""
    e = lam * np.exp(entries * np.log(100.0) / n_wn * np.arange(n_bin + 1))
    return 0.5 * (e[1:] + e[:-1]), e[1:] - e[:-1]


def test_a_large_batch_takes_no_longer_than_its_halves():
    import torch
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tables = T.XsecTables(ctx, S.make_tables(1, 1, 2, 2, 200000, with_cia=False))
    bins = T.Bins(ctx, tables, *bins_of(8, 8000, 200000))
    i0, i1 = bins.native_range
    x = torch.rand(1024, i1 - i0, dtype=torch.float64, device="cuda")

    def best(call):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ms = []
        for _ in range(8):
            a.record()
            for _ in range(20):
                call()
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b) / 20)
        return min(ms)
    whole = best(lambda: T.bin_spectra(ctx, bins, x, base=i0))
    half = best(lambda: T.bin_spectra(ctx, bins, x[:512], base=i0))
    # 0.148 ms and twice 0.075; 0.186 ms with eight lanes a bin
    assert whole <= 1.12 * 2.0 * half, (whole, half)


@pytest.mark.parametrize("n_bin,entries,B", [(8, 1270, 1030), (8, 1290, 1030), (1, 2000, 8200),
                                             (1, 2000, 16400), (3, 3060, 21850), (0, 0, 1030)])
def test_binned_spectra_are_the_oracles(n_bin, entries, B):
    import torch
    from oracle import oracle as O
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    n_wn = 40000
    tb = S.make_tables(1, 1, 2, 2, n_wn, with_cia=False)
    tables = T.XsecTables(ctx, tb)
    centre, width = bins_of(n_bin, entries, n_wn) if n_bin else bins_of(8, 30, n_wn)
    if not n_bin:                                              # one wide bin among narrow ones
        width = width.copy()
        width[3] = 0.2
    bins = T.Bins(ctx, tables, centre, width)
    i0, i1 = bins.native_range
    g = torch.Generator(device="cuda").manual_seed(B)
    flux = 0.01 + 0.01 * torch.rand(B, i1 - i0, dtype=torch.float64, device="cuda", generator=g)
    few = [0, 1, B // 2, B - 1]
    f, s = T.bin_spectra(ctx, bins, flux, flux, base=i0)
    native = np.zeros((len(few), tb.n_wn))
    native[:, i0:i1] = flux[few].cpu().numpy()
    rf, rs = O.bin_with_uncertainty(tb.wn_grid, centre, width, native, native)
    assert np.allclose(f.cpu().numpy()[few], rf, rtol=1e-12, atol=0)
    assert np.allclose(s.cpu().numpy()[few], rs, rtol=1e-12, atol=0)
    f1, _ = T.bin_spectra(ctx, bins, flux[:7].contiguous(), base=i0)     # in a small batch
    assert torch.allclose(f1, f[:7], rtol=1e-12, atol=0)
