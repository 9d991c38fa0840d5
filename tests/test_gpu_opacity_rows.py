"""The linear scheme's opacity kernel: every number of absorbers and CIA pairs it is built for,
layer counts around its 32-layer reads, steps of the brackets it treats apart (P and T steps,
diagonal steps, jumps) and ragged wavenumber counts, against the FP64 oracle (0.1 ppm, the FP32
path's bar; 1 ppm with the FP16 tables)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def tables(S, n_mol, n_cia, n_p, n_t, n_wn):
    """n_mol absorbers and n_cia pairs of the seeded recipe (beyond five absorbers: scaled copies)."""
    tb = S.make_tables(9, min(n_mol, 5), n_p, n_t, n_wn, with_cia=True)
    names, sigma = tb.species, tb.sigma
    extra = n_mol - min(n_mol, 5)
    sigma = np.concatenate([sigma] + [0.5 * sigma[k:k + 1] for k in range(extra)]).astype(np.float32)
    species = names[:5] + tuple(f"X{k}" for k in range(extra)) + names[-2:] if extra else names
    mass = np.array([S.MASS_AMU.get(s, 20.0) for s in species])
    ray = np.zeros((len(species), n_wn))
    ray[-2:] = tb.rayleigh[-2:]
    pairs = np.array([[n_mol, n_mol], [n_mol, n_mol + 1], [n_mol + 1, n_mol + 1], [0, n_mol]],
                     dtype=np.int32)[:n_cia]
    cia = np.concatenate([tb.cia, 0.25 * tb.cia])[:n_cia]
    return S.Tables(p_grid=tb.p_grid, t_grid=tb.t_grid, wn_grid=tb.wn_grid, sigma=sigma,
                    species=species, mass_amu=mass,
                    t_grid_cia=tb.t_grid_cia if n_cia else np.zeros(0),
                    cia_pair=pairs.reshape(-1, 2), cia=cia if n_cia else np.zeros((0, 0, n_wn)),
                    rayleigh=ray)


@pytest.mark.parametrize("n_mol,n_cia,n_p,n_t,n_wn,mixed", [
    (1, 0, 2, 2, 517, False), (1, 1, 13, 40, 1031, False), (2, 2, 22, 27, 1200, False),
    (3, 2, 60, 15, 769, False), (4, 0, 13, 90, 640, False), (5, 2, 13, 15, 1500, False),
    (5, 4, 22, 27, 900, False), (6, 3, 13, 15, 600, False), (8, 4, 40, 60, 523, False),
    (3, 2, 22, 60, 800, True), (8, 3, 13, 15, 600, True)])
def test_matches_the_oracle(n_mol, n_cia, n_p, n_t, n_wn, mixed):
    import torch
    from oracle import oracle as O
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tb = tables(S, n_mol, n_cia, n_p, n_t, n_wn)
    tabs = T.XsecTables(ctx, tb, storage=T.TR_STORE_FP32 | (T.TR_STORE_FP16_LOG10 if mixed else 0))
    bins_h = S.bins_logspaced(12)
    bins = T.Bins(ctx, tabs, *bins_h)
    spec_h = S.batch_spec(n_mol)
    most = 144 if mixed else 180                     # the mixed contraction's shared memory
    nl = np.array([1, 2, 9, 31, 32, 33, 64, 65, 100, most], dtype=np.int32)
    th = S.draw_theta(81, len(nl), spec_h, lx_range=(-9.0, -2.0))
    th[::2, n_mol:n_mol + 4] = [2900.0, 350.0, 2800.0, 320.0]      # steep: T jumps between layers
    spec = T.BatchSpec(spec_h, max_layers=most)
    prec = T.TR_PREC_MIXED if mixed else T.TR_PREC_FP32
    binned, status, native = T.forward_transit_batch(
        ctx, tabs, spec, torch.tensor(th, device="cuda"), torch.tensor(nl, device="cuda"), bins,
        precision=prec, native=True)
    only, st2 = T.forward_transit_batch(ctx, tabs, spec, torch.tensor(th, device="cuda"),
                                        torch.tensor(nl, device="cuda"), bins, precision=prec)
    ctx.sync_status()
    ref, st = O.forward_batch(tb, spec_h, th, nl, bins_h)
    assert np.array_equal(status.cpu().numpy(), st) and np.array_equal(st2.cpu().numpy(), st)
    tol = 1e-6 if mixed else 1e-7
    assert np.abs(binned.cpu().numpy() - ref).max() <= tol
    assert np.abs(only.cpu().numpy() - ref).max() <= tol
    assert np.isfinite(native.cpu().numpy()).all()
