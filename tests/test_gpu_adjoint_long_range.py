"""A gradient over more than 65,535 tiles of 64 wavenumbers (a binned range of 4.2 million), which
one dimension of a launch grid cannot count unless it is the first, against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_gradient_over_four_million_wavenumbers():
    import torch
    from oracle import oracle as O
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    n_wn = 4_300_000
    wn = S.wn_grid_loguniform(n_wn)
    shape = (1.0 + 0.9 * np.sin(40.0 * np.log(wn))).astype(np.float32)
    p, t = np.array([1e-5, 1e7]), np.array([300.0, 3000.0])
    sigma = np.empty((1, 2, 2, n_wn), dtype=np.float32)
    for i in range(2):
        for j in range(2):
            sigma[0, i, j] = 1e-26 * (1.0 + i + 0.5 * j) * shape
    ray = np.zeros((3, n_wn))
    ray[1] = 7.5e-49 * wn ** 4
    tb = S.Tables(p_grid=p, t_grid=t, wn_grid=wn, sigma=sigma, species=("H2O", "H2", "He"),
                  mass_amu=np.array([S.MASS_AMU[s] for s in ("H2O", "H2", "He")]),
                  t_grid_cia=np.zeros(0), cia_pair=np.zeros((0, 2), dtype=np.int32),
                  cia=np.zeros((0, 0, n_wn)), rayleigh=ray)
    ctx = T.TransitContext(0)
    tables = T.XsecTables(ctx, tb)
    bins_h = (np.array([0.9, 18.0]), np.array([1.16, 31.0]))
    bins = T.Bins(ctx, tables, *bins_h)
    i0, i1 = bins.native_range
    assert (i1 - i0) // 64 > 65535
    spec_h = S.batch_spec(1)
    spec = T.BatchSpec(spec_h, max_layers=3)
    th = np.array([[-3.0, 1500.0, 1300.0, 1100.0, 900.0, 1.0, 3.0]])
    obs, sig = np.array([0.0105, 0.0106]), np.array([5e-5, 4e-5])
    dev = lambda x: torch.tensor(x, device="cuda")
    chi2, grad, binned, status = T.adjoint_transit(ctx, tables, spec, dev(th), None, bins,
                                                   obs=dev(obs), sigma_obs=dev(sig))
    ctx.sync_status()
    assert status[0] == 0
    c, g, b, _ = O.chi2_grad(tb, spec_h, th[0], 3, bins_h, obs, sig)
    assert np.abs(binned[0].cpu().numpy() - b).max() <= 1e-7
    # the repository's bar for FP32 gradients: 1e-4, of components above a thousandth of the largest
    assert (np.abs(grad[0].cpu().numpy() - g) <= 1e-4 * np.maximum(np.abs(g), 1e-3 * np.abs(g).max())).all()
