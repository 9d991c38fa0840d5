"""The FP32 FFMA contraction with one 128-wavenumber unit per item and three K slots (layer counts
up to 120): three items of a block are in flight, so each item's path lengths need a barrier whose
earlier phases are known to be over.  Short items among the longest leave warps free to reach the
third item while the first one's path lengths arrive."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_layers,n_wn,kind", [(113, 120, 0), (120, 128, 0), (120, 97, 2),
                                                  (100, 120, 1)])
def test_one_unit_per_item_matches_the_item_alone_and_the_oracle(max_layers, n_wn, kind):
    """kind: the contraction pinned (0 the default, FFMA above 112 layers; 1, 2: 8 or 11 warps)."""
    import torch
    from oracle import oracle as O
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = S.make_tables(1, 2, 4, 5, n_wn, with_cia=False)
    tables = T.XsecTables(ctx, tb)
    spec_h = S.batch_spec(2)
    spec = T.BatchSpec(spec_h, max_layers=max_layers)
    B = 1400
    th_h = S.draw_theta(31, B, spec_h)
    nl_h = np.random.default_rng(max_layers).integers(1, 61, B).astype(np.int32)
    nl_h[::9] = max_layers
    nl_h[4::31] = 1
    th_h[7, 0] = 1.0                                                # sum X > 1: rejected
    th, nl = torch.tensor(th_h, device="cuda"), torch.tensor(nl_h, device="cuda")

    def pin(b):
        if kind:
            T.pin_forward_config(ctx, tables, spec, b, None, native=True, contract_per_sm=kind)
    pin(B)
    pin(1)
    first = status = None
    for _ in range(40):
        _, st, native = T.forward_transit_batch(ctx, tables, spec, th, nl, None, native=True)
        first, status = (native.clone(), st) if first is None else (first, status)
        assert torch.equal(native, first)
    ctx.sync_status()
    for b in range(0, B, 7):
        _, st, alone = T.forward_transit_batch(ctx, tables, spec, th[b:b + 1].contiguous(),
                                               nl[b:b + 1].contiguous(), None, native=True)
        assert st[0] == status[b] and torch.equal(alone[0], first[b]), b
    ctx.sync_status()
    assert status[7] == T.TR_ERR_INVALID_MODEL
    for b in (b for b in (0, 1, 2, 9, 700, 1398, 1399) if status[b] == 0):
        m, nt = spec_h.n_mol, spec_h.n_tnodes
        atm = S.Atmosphere(n_layers=int(nl_h[b]), p_max=spec_h.p_max, p_min=spec_h.p_min,
                           tnode_log10p=spec_h.tnode_log10p, tnode_t=th_h[b, m:m + nt],
                           log10_x=th_h[b, :m], fill_frac=spec_h.fill_frac,
                           r_p=th_h[b, m + nt] * S.R_JUP, m_p=spec_h.m_p, r_s=spec_h.r_s,
                           p_cloud_top=10.0 ** th_h[b, m + nt + 1], p_cloud_bot=spec_h.p_cloud_bot,
                           kappa_cloud=spec_h.kappa_cloud, gravity_mode=spec_h.gravity_mode,
                           cloud_mode=spec_h.cloud_mode)
        assert np.abs(first[b].cpu().numpy() - O.forward(tb, atm)[0]).max() <= 1e-7, b
