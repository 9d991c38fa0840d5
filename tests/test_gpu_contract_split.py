"""The FP32 contraction for more than 112 layers divides a batch's units among the blocks by cost
(layer counts differ): every item of a batch equals, bit for bit, the item alone, for batches of
fewer items than threads, more, an invalid item and items of one layer among the longest."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_wn", [(2, 20000), (19, 3000), (153, 300), (700, 260)])
def test_items_of_a_batch_equal_the_item_alone(B, n_wn):
    import torch
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(1, 2, 4, 5, n_wn, with_cia=False)
    tables = T.XsecTables(ctx, tb)
    spec_h = S.batch_spec(2)
    spec = T.BatchSpec(spec_h, max_layers=150)
    th = torch.tensor(S.draw_theta(5, B, spec_h), device="cuda")
    rng = np.random.default_rng(B)
    nl_h = rng.choice([1, 2, 16, 17, 64, 113, 149, 150], B).astype(np.int32)
    nl_h[0], nl_h[-1] = 150, 1
    if B > 2:
        th[1, 0] = 1.0                                          # sum X > 1: rejected
    nl = torch.tensor(nl_h, device="cuda")
    _, status, native = T.forward_transit_batch(ctx, tables, spec, th, nl, None, native=True)
    ctx.sync_status()
    for b in sorted({0, 1, 2 % B, B // 2, (B // 2 + 1) % B, B - 2, B - 1}):
        _, st, alone = T.forward_transit_batch(ctx, tables, spec, th[b:b + 1].contiguous(),
                                               nl[b:b + 1].contiguous(), None, native=True)
        assert st[0] == status[b] and torch.equal(alone[0], native[b]), b
    ctx.sync_status()
