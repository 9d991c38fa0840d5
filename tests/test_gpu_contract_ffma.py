"""The FP32 FFMA contraction (layer counts above 112): an item's second 128-wavenumber unit may
be ready before the item's path lengths have landed, so every warp waits for both."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [17, 40, 113])
def test_repeated_batches_are_bitwise_equal_and_match_the_oracle(layers):
    """Items with few ray tiles leave warps free to start on the next unit while the first
    unit's loads are in flight; two units per item, several items per CTA."""
    import torch
    from oracle import oracle as O
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(1, 2, 13, 15, 3000, with_cia=False)
    tables = T.XsecTables(ctx, tb)
    bins = T.Bins(ctx, tables, *S.bins_logspaced(20))
    spec_h = S.batch_spec(2)
    B = 912
    spec = T.BatchSpec(spec_h, max_layers=150)
    th_h = S.draw_theta(71, B, spec_h)
    nl_h = np.full(B, layers, dtype=np.int32)
    nl_h[5::7] = 150
    th, nl = torch.tensor(th_h, device="cuda"), torch.tensor(nl_h, device="cuda")
    first = None
    for _ in range(40):
        binned, status = T.forward_transit_batch(ctx, tables, spec, th, nl, bins)
        first = binned.clone() if first is None else first
        assert torch.equal(binned, first)
    ctx.sync_status()
    pick = [0, 1, 5, 6, 455, 456, 910, 911]
    ref, st = O.forward_batch(tb, spec_h, th_h[pick], nl_h[pick], S.bins_logspaced(20))
    assert np.array_equal(status.cpu().numpy()[pick], st)
    assert np.abs(first.cpu().numpy()[pick] - ref).max() <= 1e-7
