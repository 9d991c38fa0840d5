"""The adjoint's tile kernel at the edges of its layer tiles (8 layers), of the shared memory that lets
three blocks share an SM (101 layers) or two, with one to five absorbers, and
with and without species that have no Rayleigh cross-sections.

Bar: against the FP64 oracle's exact gradient, |g - g_ref| <= 1e-4 max(|g_ref|, 1e-3 max|g_ref|)
per component, the bar of the adjoint's other tests."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1912_07759_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mol,with_cia,with_ray,most,layers", [
    (5, True, True, 101, [1, 8, 9, 101]),
    (5, False, True, 104, [7, 97, 104]),
    (1, True, False, 150, [16, 129, 150]),
    (5, True, True, 24, [2, 17, 24]),
    (2, False, False, 33, [32, 33]),
])
def test_gradient_at_tile_edges(n_mol, with_cia, with_ray, most, layers):
    import torch
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(60 + n_mol, n_mol, 13, 15, 1200, with_cia=with_cia, with_rayleigh=with_ray,
                       wn_min=4000.0, wn_max=12000.0)
    tables = T.XsecTables(ctx, tb)
    bins_h = S.bins_logspaced(6, 1.2, 1.6)
    bins = T.Bins(ctx, tables, *bins_h)
    spec_h = S.batch_spec(n_mol)
    B = len(layers)
    th = S.draw_theta(23, B, spec_h, lx_range=(-6.0, -2.5), t_range=(900.0, 1900.0),
                      lpc_range=(2.5, 4.5))
    gbin = np.random.default_rng(3).normal(size=(B, len(bins_h[0])))
    _, grad, _, status = T.adjoint_transit(
        ctx, tables, T.BatchSpec(spec_h, max_layers=most), torch.tensor(th, device="cuda"),
        torch.tensor(np.array(layers, dtype=np.int32), device="cuda"), bins,
        gbin=torch.tensor(gbin, device="cuda"))
    assert not status.any()
    ctx.sync_status()
    one = np.ones(len(bins_h[0]))
    for b, n in enumerate(layers):
        jac = O.chi2_grad(tb, spec_h, th[b], n, bins_h, 0 * one, one)[3]
        g, ref = grad[b].cpu().numpy(), gbin[b] @ jac
        floor = 1e-3 * np.abs(ref).max()
        assert (np.abs(g - ref) <= 1e-4 * np.maximum(np.abs(ref), floor)).all(), (n, g, ref)


def test_tile_sums_of_a_large_batch_equal_a_small_one():
    """The tile sums of launches large enough take four elements a thread, features one at a time
    where a slot's are not a multiple of four (33 layers of 9): the same sums, bit for bit."""
    import torch
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(5, 2, 4, 5, 3000, with_cia=False)
    tables = T.XsecTables(ctx, tb)
    bins_h = S.bins_logspaced(6)
    bins = T.Bins(ctx, tables, *bins_h)
    spec_h = S.batch_spec(2)
    B = 1500
    spec = T.BatchSpec(spec_h, max_layers=33)
    th = torch.tensor(S.draw_theta(41, B, spec_h), device="cuda")
    nl = torch.tensor(np.random.default_rng(1).integers(1, 34, B).astype(np.int32), device="cuda")
    gbin = torch.tensor(np.random.default_rng(2).normal(size=(B, 6)), device="cuda")
    _, grad, _, _ = T.adjoint_transit(ctx, tables, spec, th, nl, bins, gbin=gbin, want_binned=False)
    for b in (0, 700, 1488):
        part = slice(b, b + 12)
        _, g, _, _ = T.adjoint_transit(ctx, tables, spec, th[part].contiguous(), nl[part].contiguous(),
                                       bins, gbin=gbin[part].contiguous(), want_binned=False)
        assert torch.equal(g, grad[part]), b
    ctx.sync_status()
