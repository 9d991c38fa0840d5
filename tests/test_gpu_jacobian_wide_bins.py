"""A Jacobian of wide bins (each of more than 256 tiles of 64 wavenumbers) takes each bin's own
tiles, not the whole range once per bin: its tile kernel's time is about one gradient's, and its
rows equal the vector-Jacobian products with the bins' unit vectors."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_each_row_takes_its_own_tiles():
    import torch
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tables = T.XsecTables(ctx, S.make_tables(6, 1, 2, 3, 200000, with_cia=False))
    bins = T.Bins(ctx, tables, *S.bins_logspaced(8, 0.4, 14.0))
    assert (bins.native_range[1] - bins.native_range[0]) // (8 * 64) > 256
    spec_h = S.batch_spec(1)
    spec = T.BatchSpec(spec_h, max_layers=24)
    th = torch.tensor(S.draw_theta(2, 2, spec_h, lx_range=(-8.0, -3.0)), device="cuda")
    unit = torch.zeros(2, 8, dtype=torch.float64, device="cuda")

    def jacobian():
        return T.adjoint_transit(ctx, tables, spec, th, None, bins, want_grad=False, want_jac=True,
                                 want_binned=False)[4]

    def product():
        return T.adjoint_transit(ctx, tables, spec, th, None, bins, gbin=unit, want_binned=False)[1]
    jac = jacobian()
    for k in range(8):
        unit.zero_()
        unit[:, k] = 1.0
        g = product()
        scale = g.abs().amax(dim=1, keepdim=True).clamp_min(1e-300)
        # the same FP32 terms and tile sums; FP64 sums of about 1e2 terms: 1e-13
        assert ((jac[:, k] - g).abs() / scale).max().item() <= 1e-13
    ms = {}
    for name, call in (("product", product), ("jacobian", jacobian)):
        T.profile_enable(ctx)
        for _ in range(10):
            call()
        torch.cuda.synchronize()
        ms[name] = T.profile_read(ctx)["k_adjoint_tile"][0]
    T.profile_enable(ctx, False)
    assert ms["jacobian"] <= 3.0 * ms["product"], ms       # eight times when each takes the range
    ctx.sync_status()
