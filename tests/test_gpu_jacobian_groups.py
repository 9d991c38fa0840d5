"""The Jacobian's rows are done in groups of wavenumber tiles: every row equals the vector-Jacobian
product with that bin's unit vector (a separate pass over all tiles), for bins within one tile,
bins over several tiles, more rows than one group holds, overlapping bins, and a bin of more tiles
than a group can list."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_wn,centre,width", [
    (3000, None, None),                                        # narrow bins, several groups
    (40000, [1.15, 1.2, 1.21, 1.6], [0.08, 0.02, 0.3, 0.001]),   # overlapping, wide and narrow
    (200000, [1.4, 1.2, 1.65], [0.6, 0.01, 0.05]),               # the first has 296 tiles
])
def test_rows_equal_unit_products(n_wn, centre, width):
    import torch
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(5, 2, 3, 4, n_wn, with_cia=True)
    tables = T.XsecTables(ctx, tb)
    c, w = S.bins_logspaced(40) if centre is None else (np.array(centre), np.array(width))
    bins = T.Bins(ctx, tables, c, w)
    spec_h = S.batch_spec(2)
    B = 3
    spec = T.BatchSpec(spec_h, max_layers=33)
    th = torch.tensor(S.draw_theta(17, B, spec_h, lx_range=(-9.0, -3.0)), device="cuda")
    th[1, 0] = 1.0                                             # sum X > 1: a rejected item
    nl = torch.tensor([33, 20, 1], dtype=torch.int32, device="cuda")
    _, _, _, status, jac = T.adjoint_transit(ctx, tables, spec, th, nl, bins, want_grad=False,
                                             want_jac=True)
    assert status.tolist() == [0, T.TR_ERR_INVALID_MODEL, 0]
    assert not jac[1].any()
    for k in sorted({0, 1, len(c) // 2, len(c) - 1}):
        e = torch.zeros(B, len(c), dtype=torch.float64, device="cuda")
        e[:, k] = 1.0
        _, g, _, _ = T.adjoint_transit(ctx, tables, spec, th, nl, bins, gbin=e, want_binned=False)
        scale = g.abs().amax(dim=1, keepdim=True).clamp_min(1e-300)
        # the same FP32 terms and tile sums; FP64 sums of about 1e2 terms: 1e-13
        assert ((jac[:, k] - g).abs() / scale).max().item() <= 1e-13
    ctx.sync_status()
