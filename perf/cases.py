"""The calls a user of the framework makes, as cases to time and to compare: single forward
models, sampler batches, chi^2 gradients, Jacobians, emission spectra and simulated
observations, through the public entry points of `paper_1912_07759_gb300`.

A case is a dict of plain values.  `prepare` makes its inputs from a seed (parameter vectors,
observations, noise draws) and the handles a program keeps (context, tables, bins); the tables
of one shape are loaded once per process and shared, as a program loads its cross-sections
once.  `run` is one pass; `exact` states the same outputs in 64-bit torch, independent of the
framework's code.
"""
import collections
import functools
import math

import numpy as np
import torch

from paper_1912_07759_gb300 import synthetic as S
from paper_1912_07759_gb300 import transit as T

G_NEWTON, K_BOLTZ, AMU = 6.67430e-11, 1.380649e-23, 1.66053906660e-27
HC_K = 6.62607015e-34 * 299792458.0 / K_BOLTZ * 100.0      # h c / k_B per cm^-1
LN10 = math.log(10.0)
T_STAR = 5800.0
SNR, N_OBS = 200.0, 4

# Every case carries all of these.  kind: which call; items: atmospheres (spectra for
# "instrument"); layers: the largest layer count; uneven: layer counts drawn from a third of it
# up; wavenumbers: native grid; p, t: table grid; mixed: FP16 tables and the mixed path; exp: the
# exponential temperature scheme; profiles: Guillot temperatures and two-layer gases.
DEFAULTS = dict(items=1, layers=100, uneven=False, wavenumbers=10000, absorbers=2, p=13, t=15,
                cia=True, bins=50, mixed=False, exp=False, profiles=False, angles=4)


def _case(name, kind, **kw):
    return dict(DEFAULTS, name=name, kind=kind, **kw)


def listed():
    return [
        # one model built from a description and evaluated once, at the paper's R = 10,000 over
        # 0.3-15 um, 100 layers, two absorbers: what an interactive user or a script does
        _case("one_model", "model", wavenumbers=39121),
        # a sampler's likelihood call for one live point: the smallest call
        _case("live_point", "binned", cia=False),
        # the full-size model, replayed as a graph with new parameters each time (native + bins)
        _case("full_size_graph", "graph", wavenumbers=200000, absorbers=5, p=22, t=27),
        # thousands of live points at once, uneven layer counts
        _case("live_points_4096", "binned", items=4096, layers=150, uneven=True, cia=False),
        # a grid of full-size native spectra (model libraries, training sets)
        _case("spectra_64", "spectra", items=64, wavenumbers=200000, absorbers=5, p=22, t=27),
        # the same through the mixed-precision path
        _case("spectra_mixed_32", "spectra", items=32, wavenumbers=200000, absorbers=5, p=22,
              t=27, mixed=True),
        # chi^2 and its gradient for a few chains of a gradient-based sampler
        _case("gradient_8", "gradient", items=8, wavenumbers=39121, absorbers=5),
        # many chains at low resolution: the opacities stay in the workspace
        _case("gradient_1024", "gradient", items=1024, absorbers=5, cia=False),
        # many chains on the full-size tables: the opacities outgrow the workspace
        _case("gradient_full_320", "gradient", items=320, wavenumbers=200000, absorbers=5, p=22,
              t=27),
        # Jacobians for Fisher matrices
        _case("jacobian_128", "jacobian", items=128, absorbers=5, cia=False),
        # one full-size eclipse spectrum
        _case("emission", "emission", wavenumbers=200000, absorbers=5, p=22, t=27),
        # simulated observations: binning with uncertainties, then the instrument's noise
        _case("instrument_1024", "instrument", items=1024, wavenumbers=200000),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds with sizes spread over their ranges."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["model", "binned", "binned", "graph", "spectra", "spectra",
                           "gradient", "gradient", "jacobian", "emission", "instrument"])
        wn = _log_uniform(rng, 2000, 200000)
        c = dict(DEFAULTS, kind=kind, wavenumbers=wn, absorbers=rng.randint(1, 5),
                 layers=rng.randint(20, 150), p=rng.randint(10, 22), t=rng.randint(10, 27),
                 cia=rng.random() < 0.7, bins=rng.randint(10, 60))
        if kind not in ("model", "graph", "emission"):
            c["items"] = _log_uniform(rng, 1, 4096)
            c["uneven"] = kind != "instrument" and rng.random() < 0.5
        if kind == "emission":
            c["items"] = _log_uniform(rng, 1, 32)
            c["angles"] = rng.choice([2, 4, 8])
        if kind in ("graph", "spectra", "gradient"):
            c["mixed"] = rng.random() < 0.2
        if kind in ("binned", "spectra") and rng.random() < 0.15:
            c["exp"] = True
        elif kind in ("binned", "spectra", "emission") and rng.random() < 0.15:
            c["profiles"] = True
        if _cost(c) <= most:
            return c


# ------------------------------------------------------------------------------------ work
def _binned_wavenumbers(c):
    return max(1, int(c["wavenumbers"] * math.log(1.7 / 1.1) / math.log(100.0)))


def work(c):
    """What one pass cannot do without.  Table rows: an atmosphere crosses about three (P, T)
    rows per table pressure; many together touch at most all of them."""
    B, N, M, nb = c["items"], c["layers"], c["absorbers"], c["bins"]
    n_in = _binned_wavenumbers(c)
    if c["kind"] == "instrument":
        return {"bytes": 16.0 * B * n_in + 48.0 * B * nb, "flops": 5.0 * B * n_in}
    W = n_in if c["kind"] in ("binned", "gradient", "jacobian") else c["wavenumbers"]
    if c["uneven"]:
        N = 2 * N / 3                                       # mean of N/3 .. N
    rows = min(c["p"] * c["t"], 3 * c["p"] * B)
    read = rows * M * W * (2.0 if c["mixed"] else 4.0)
    read += (2 * min(c["t"], 16 * B) * W * 4.0 if c["cia"] else 0.0) + 2 * W * 4.0
    theta = M + 6
    wrote = {"model": W + nb, "graph": W + nb, "spectra": B * (W + nb), "emission": B * (W + nb),
             "binned": B * nb, "gradient": B * (nb + theta + 1), "jacobian": B * nb * theta}
    cell = 16.0 + 8.0 * M * (5 if c["exp"] else 0.3)         # opacity of one layer, wavenumber
    column = N * (N + 1) + 4.0 * N                           # optical depths and their sum
    if c["kind"] == "emission":
        column = N * (4.0 + 4.0 * c["angles"])
    if c["kind"] in ("gradient", "jacobian"):
        column *= 3.0
        cell += 8.0 * M + 10.0
    return {"bytes": read + 8.0 * wrote[c["kind"]], "flops": B * W * (N * cell + column)}


def _cost(c):
    w = work(c)
    return w["flops"] + 10.0 * w["bytes"]


# ---------------------------------------------------------------------------------- inputs
def _table_key(c):
    return (c["absorbers"], c["p"], c["t"], c["wavenumbers"], c["cia"], c["exp"])


@functools.lru_cache(maxsize=2)
def _host_tables(n_mol, n_p, n_t, n_wn, cia, exp):
    """Synthetic cross-sections of the package's recipe (10^x taken on the GPU where there is
    one: the full-size tables hold 594 M values)."""
    p_grid = np.exp(np.linspace(math.log(1e-5), math.log(1e7), n_p))
    t_grid = np.linspace(300.0, 3000.0, n_t)
    wn = S.wn_grid_loguniform(n_wn)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    sigma = np.empty((n_mol, n_p, n_t, n_wn), dtype=np.float32)
    for m in range(n_mol):
        lx = torch.from_numpy(S.log10_xsec_cm2(2000 + m, p_grid, t_grid, wn)).to(dev) - 4.0
        sigma[m] = torch.pow(10.0, lx).cpu().numpy()
    base = S.make_tables(2, 1, 2, n_t, n_wn, with_cia=cia)   # CIA, Rayleigh of the recipe
    species = tuple(S.ABSORBERS[:n_mol]) + ("H2", "He")
    ray = np.zeros((n_mol + 2, n_wn))
    ray[n_mol:] = base.rayleigh[1:]
    return S.Tables(p_grid=p_grid, t_grid=t_grid, wn_grid=wn, sigma=sigma, species=species,
                    mass_amu=np.array([S.MASS_AMU[s] for s in species]),
                    t_grid_cia=base.t_grid_cia,
                    cia_pair=(base.cia_pair + (n_mol - 1)).astype(np.int32), cia=base.cia,
                    rayleigh=ray, interp_mode=S.INTERP_EXP if exp else S.INTERP_LINEAR)


_loaded = collections.OrderedDict()


def _context():
    if "ctx" not in _loaded:
        _loaded["ctx"] = T.TransitContext(0)
    return _loaded["ctx"]


def _loaded_tables(c):
    """The tables' handle; the last three shapes stay loaded."""
    key = _table_key(c) + (c["mixed"],)
    if key not in _loaded:
        storage = T.TR_STORE_FP32 | (T.TR_STORE_FP16_LOG10 if c["mixed"] else 0)
        _loaded[key] = T.XsecTables(_context(), _host_tables(*_table_key(c)), storage=storage)
        for old in [k for k in _loaded if k != "ctx"][:-3]:
            del _loaded[old]
    return _loaded[key]


def _spec(c):
    spec = S.batch_spec(c["absorbers"])
    if c["kind"] in ("model", "graph", "emission"):
        spec.cloud_mode = S.CLOUD_DISCRETE
    if c["profiles"]:
        spec.t_profile, spec.gas_mode = S.TPROF_GUILLOT, S.GAS_TWOLAYER
    return spec


def _host_inputs(c, seed):
    """theta [items][n_theta], layer counts, observation and its uncertainties."""
    spec = _spec(c)
    rng = np.random.default_rng(seed)
    if c["kind"] in ("model", "graph", "emission") and not c["profiles"]:
        # around the full-size model: hot below, cool above, cloud top near 1e3 Pa
        n = c["items"]
        th = np.concatenate([rng.uniform(-8.0, -3.0, (n, c["absorbers"])),
                             np.array([2200.0, 1700.0, 1200.0, 800.0]) + rng.uniform(-150.0, 150.0, (n, 4)),
                             rng.uniform(0.9, 1.1, (n, 1)), rng.uniform(2.5, 3.5, (n, 1))], axis=1)
    else:
        th = S.draw_theta(seed + 1, c["items"], spec)
    nl = np.full(c["items"], c["layers"], dtype=np.int32)
    if c["uneven"]:
        nl = S.draw_nlayers(seed + 2, c["items"], max(1, c["layers"] // 3), c["layers"])
    sig, z = S.obs_noise(seed + 3, c["bins"])
    return spec, th, nl, 0.0105 + sig * z, sig


def _instrument_inputs(c, seed, n, dev):
    g = torch.Generator(device=dev).manual_seed(seed)
    rand = dict(dtype=torch.float64, device=dev, generator=g)
    flux = 0.0105 + 1e-4 * torch.randn(c["items"], n, **rand)
    sigma = 3e-5 * (1.0 + torch.rand(c["items"], n, **rand))
    return flux, sigma, torch.randn(c["items"], c["bins"], **rand)


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.ctx, s.tables = case, _context(), _loaded_tables(case)
    s.bins = T.Bins(s.ctx, s.tables, *S.bins_logspaced(case["bins"]))
    dev = torch.device("cuda", 0)
    s.precision = T.TR_PREC_MIXED if case["mixed"] else T.TR_PREC_FP32
    if case["kind"] == "instrument":
        i0, i1 = s.bins.native_range
        s.base = i0
        s.flux, s.sigma, s.z = _instrument_inputs(case, seed, i1 - i0, dev)
        return s
    spec, th, nl, obs, sig = _host_inputs(case, seed)
    if case["kind"] == "model":
        s.atm = _description(case, spec, th[0], nl[0])
        return s
    s.spec = T.BatchSpec(spec, max_layers=case["layers"])
    s.theta = torch.tensor(th, device=dev)
    s.nlayers = torch.tensor(nl, device=dev) if case["uneven"] else None
    s.obs, s.sig = torch.tensor(obs, device=dev), torch.tensor(sig, device=dev)
    native = case["kind"] in ("graph", "spectra", "emission")
    s.workspace = torch.empty(
        T.batch_workspace_size(s.ctx, s.tables, s.spec, None if native else s.bins, case["items"],
                               with_adjoint=case["kind"] in ("gradient", "jacobian")),
        dtype=torch.uint8, device=dev)
    if case["kind"] == "graph":
        s.graph = T.ForwardGraph(s.ctx, s.tables, s.spec, s.theta.clone(), s.nlayers, s.bins,
                                 precision=s.precision, workspace=s.workspace, native=True,
                                 autotune=False)
    return s


def _description(case, spec, th, layers):
    m, nt = spec.n_mol, spec.n_tnodes
    return S.Atmosphere(n_layers=int(layers), p_max=spec.p_max, p_min=spec.p_min,
                        tnode_log10p=spec.tnode_log10p, tnode_t=th[m:m + nt], log10_x=th[:m],
                        fill_frac=spec.fill_frac, r_p=th[m + nt] * S.R_JUP, m_p=spec.m_p,
                        r_s=spec.r_s, p_cloud_top=10.0 ** th[m + nt + 1],
                        kappa_cloud=spec.kappa_cloud, gravity_mode=spec.gravity_mode,
                        cloud_mode=spec.cloud_mode)


def run(s):
    kind = s.case["kind"]
    if kind == "model":
        atm = T.Atmosphere(s.ctx, s.tables, s.atm)
        native, binned = T.forward_transit(s.ctx, s.tables, atm, s.bins, precision=s.precision)
        return {"native": native, "binned": binned}
    if kind == "graph":
        s.graph.theta.copy_(s.theta)
        s.graph.launch()
        return {"native": s.graph.native, "binned": s.graph.binned, "status": s.graph.status}
    if kind == "binned":
        binned, status = T.forward_transit_batch(s.ctx, s.tables, s.spec, s.theta, s.nlayers,
                                                 s.bins, workspace=s.workspace)
        return {"binned": binned, "status": status}
    if kind == "spectra":
        binned, status, native = T.forward_transit_batch(
            s.ctx, s.tables, s.spec, s.theta, s.nlayers, s.bins, precision=s.precision,
            workspace=s.workspace, native=True)
        return {"native": native, "binned": binned, "status": status}
    if kind == "gradient":
        chi2, grad, binned, status = T.adjoint_transit(
            s.ctx, s.tables, s.spec, s.theta, s.nlayers, s.bins, obs=s.obs, sigma_obs=s.sig,
            precision=s.precision, workspace=s.workspace)
        return {"chi2": chi2, "grad": grad, "binned": binned, "status": status}
    if kind == "jacobian":
        _, _, binned, status, jac = T.adjoint_transit(
            s.ctx, s.tables, s.spec, s.theta, s.nlayers, s.bins, workspace=s.workspace,
            want_grad=False, want_jac=True)
        return {"binned": binned, "jac": jac, "status": status}
    if kind == "emission":
        binned, status, native = T.forward_emission_batch(
            s.ctx, s.tables, s.spec, s.theta, s.nlayers, s.bins, n_mu=s.case["angles"],
            t_star=T_STAR, native=True, workspace=s.workspace)
        return {"native": native, "binned": binned, "status": status}
    binned, binned_sigma = T.bin_spectra(s.ctx, s.bins, s.flux, s.sigma, base=s.base)
    obs, noise = T.snr_instrument(s.ctx, binned, SNR, N_OBS, s.z)
    return {"binned": binned, "binned_sigma": binned_sigma, "obs": obs, "noise": noise}


# ------------------------------------------------------------------------ 64-bit statement
def _bin_matrix(c, dev):
    """Overlap weights [i1 - i0][bins] of the native bins (midpoint edges) and the range."""
    wn = S.wn_grid_loguniform(c["wavenumbers"])
    mid = 0.5 * (wn[1:] + wn[:-1])
    edge = np.concatenate([[wn[0] - 0.5 * (wn[1] - wn[0])], mid, [wn[-1] + 0.5 * (wn[-1] - wn[-2])]])
    lo, hi = 1e4 / edge[1:], 1e4 / edge[:-1]
    centre, width = S.bins_logspaced(c["bins"])
    bm, bp = centre - 0.5 * width, centre + 0.5 * width
    i = np.nonzero((hi > bm.min()) & (lo < bp.max()))[0]
    i0, i1 = int(i[0]), int(i[-1]) + 1
    ov = np.minimum(bp, hi[i0:i1, None]) - np.maximum(bm, lo[i0:i1, None])
    w = np.where(ov > 0.0, ov / (hi - lo)[i0:i1, None], 0.0)
    return torch.tensor(w, device=dev), i0, i1


class _Model:
    """The discrete forward model of a case in float64 torch, differentiable in theta."""

    def __init__(self, c, seed):
        self.c = c
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.spec, self.th, self.nl, self.obs, self.sig = _host_inputs(c, seed)
        tb = _host_tables(*_table_key(c))
        self.n_mol = tb.n_mol
        self.d = lambda x: torch.tensor(np.asarray(x), dtype=torch.float64, device=self.dev)
        self.sigma = torch.from_numpy(tb.sigma).to(self.dev)
        self.pg, self.tg, self.wn = self.d(tb.p_grid), self.d(tb.t_grid), self.d(tb.wn_grid)
        self.cia, self.ray = self.d(tb.cia), self.d(tb.rayleigh)
        self.pairs, self.mass = tb.cia_pair.tolist(), self.d(tb.mass_amu)

    @staticmethod
    def axis(grid, x):
        xc = torch.minimum(torch.maximum(x, grid[0]), grid[-1])
        i = (torch.searchsorted(grid, xc.detach().contiguous(), right=True) - 1).clamp(0, grid.numel() - 2)
        return i, (xc - grid[i]) / (grid[i + 1] - grid[i])

    @staticmethod
    def e2(x):
        """E_2 = e^-x - x E_1: series of E_1 up to 2, its continued fraction beyond."""
        xs, xl = x.clamp(max=2.0), x.clamp(min=2.0)
        s, term = torch.zeros_like(x), torch.ones_like(x)
        for k in range(1, 60):
            term = term * (-xs / k)
            s = s - term / k
        small = -0.57721566490153286061 - torch.log(xs) + s
        t = torch.zeros_like(x)
        for k in range(400, 0, -1):
            t = k / (1.0 + k / (xl + t))
        e1 = torch.where(x <= 2.0, small, torch.exp(-xl) / (xl + t))
        return torch.exp(-x) - x * e1

    def profile(self, th, nl):
        """Layer quantities [b][N] of the items (N the largest count; layers beyond an item's
        own carry no path length and no annulus)."""
        sp, M = self.spec, self.n_mol
        nl = torch.tensor(nl, device=self.dev, dtype=torch.float64)[:, None]
        N = int(nl.max())
        l = torch.arange(N + 1, device=self.dev, dtype=torch.float64)[None]
        lmax, lmin = math.log(sp.p_max), math.log(sp.p_min)
        lb = lmax + (lmin - lmax) * l / nl                  # ln p of the boundaries
        delta = (lmax - lmin) / nl
        lnp = 0.5 * (lb[:, 1:] + lb[:, :-1])
        P = torch.exp(lnp)
        k = sp.n_chem
        rp, lpc = th[:, k + sp.n_tpar, None] * S.R_JUP, th[:, k + sp.n_tpar + 1, None]
        gm = G_NEWTON * sp.m_p
        if sp.t_profile == S.TPROF_GUILLOT:
            def temperature(p):
                g = th[:, k:k + 5]
                kir = torch.pow(10.0, g[:, 1:2])
                tau = kir * p / (gm / rp ** 2)
                out = 0.75 * sp.t_int ** 4 * (2.0 / 3.0 + tau)
                for j, wgt in ((2, 1.0 - g[:, 4:5]), (3, g[:, 4:5])):
                    gm_j = torch.pow(10.0, g[:, j:j + 1]) / kir
                    gt = gm_j * tau
                    xi = (2.0 / 3.0 + 2.0 / (3.0 * gm_j) * (1.0 + (gt / 2.0 - 1.0) * torch.exp(-gt))
                          + 2.0 * gm_j / 3.0 * (1.0 - tau ** 2 / 2.0) * self.e2(gt))
                    out = out + 0.75 * g[:, 0:1] ** 4 * wgt * xi
                return out ** 0.25
        else:
            node = self.d(sp.tnode_log10p[::-1].copy())     # ascending
            tn = th[:, k:k + sp.n_tnodes].flip(1)

            def temperature(p):
                i, f = self.axis(node, (torch.log(p) / LN10).expand(th.shape[0], -1))
                a, b = tn.gather(1, i), tn.gather(1, i + 1)
                return a + (b - a) * f
        temp = temperature(P)
        t_surf = temperature(torch.full_like(P[:, :1], sp.p_max))
        x = torch.pow(10.0, th[:, :M])[:, None, :].expand(-1, N, -1)
        if sp.gas_mode == S.GAS_TWOLAYER:
            top = torch.pow(10.0, th[:, M:2 * M])[:, None, :]
            sw = th[:, None, 2 * M:3 * M] * LN10
            f = ((lb[:, :-1, None] - torch.maximum(sw, lb[:, 1:, None])) / delta[:, :, None]).clamp(0.0, 1.0)
            x = f * x + (1.0 - f) * top
        fill = self.d(sp.fill_frac)
        x = torch.cat([x, (1.0 - x.sum(-1, keepdim=True)) * fill], dim=-1)
        mu = x @ self.mass
        z = [torch.zeros_like(rp)]
        for j in range(N):
            step = K_BOLTZ * temp[:, j:j + 1] * delta / (mu[:, j:j + 1] * AMU * gm) * (rp + z[-1]) ** 2
            z.append(z[-1] + step)
        z = torch.cat(z, dim=1)
        rho = P / (K_BOLTZ * temp)
        inside = l[:, :-1] < nl
        if sp.cloud_mode == S.CLOUD_DISCRETE:
            cloud = ((P >= torch.pow(10.0, lpc)) & (P <= sp.p_max)).double()
        else:
            cloud = ((lb[:, :-1] - torch.maximum(lpc * LN10, lb[:, 1:])) / delta).clamp(0.0, 1.0)
        return dict(P=P, T=temp, X=x, rho=rho, z=z, rp=rp, cloud=cloud, inside=inside, t_surf=t_surf)

    def opacity(self, f, i0, i1):
        """K [b][N][i1 - i0]."""
        N = f["T"].shape[1]
        ip, tp = self.axis(self.pg, f["P"])
        it, tt = self.axis(self.tg, f["T"])
        tp, tt = tp[..., None], tt[..., None]
        K = (self.spec.kappa_cloud * f["cloud"])[..., None].expand(-1, N, i1 - i0)
        K = K + (f["rho"][..., None] * f["X"]) @ self.ray[:, i0:i1]
        for m in range(self.n_mol):
            tab = self.sigma[m, :, :, i0:i1]
            c = [tab[ip + a, it + b].double() for a in (0, 1) for b in (0, 1)]
            if self.c["exp"]:
                T1, T2 = self.tg[it][..., None], self.tg[it + 1][..., None]
                Tc = T1 + tt * (T2 - T1)
                u = (1.0 / T1 - 1.0 / Tc) / (1.0 / T1 - 1.0 / T2)
                lo, hi = (torch.exp(torch.log(c[a]) * (1.0 - u) + torch.log(c[a + 1]) * u) for a in (0, 2))
            else:
                lo, hi = c[0] + (c[1] - c[0]) * tt, c[2] + (c[3] - c[2]) * tt
            K = K + (f["rho"] * f["X"][..., m])[..., None] * (lo + (hi - lo) * tp)
        for q, (a, b) in enumerate(self.pairs):
            w = f["rho"] ** 2 * f["X"][..., a] * f["X"][..., b]
            tab = self.cia[q, :, i0:i1]
            K = K + w[..., None] * (tab[it] + (tab[it + 1] - tab[it]) * tt)   # same T grid
        return K

    def depth(self, f, i0, i1):
        """Transit depth [b][i1 - i0]."""
        z, rp = f["z"], f["rp"]
        N = z.shape[1] - 1
        d = z[:, None, :] - z[:, :N, None]                   # z_k - z_j  [b][j][k]
        up = torch.arange(N + 1, device=self.dev)[None, :] > torch.arange(N, device=self.dev)[:, None]
        s2 = torch.where(up, d * (2.0 * rp[..., None] + z[:, None, :] + z[:, :N, None]), torch.ones_like(d))
        s = torch.where(up, torch.sqrt(s2), torch.zeros_like(d))
        DL = 2.0 * (s[:, :, 1:] - s[:, :, :-1]) * f["inside"][:, None, :]
        A = (z[:, 1:] - z[:, :-1]) * (2.0 * rp + z[:, 1:] + z[:, :-1]) * f["inside"]
        tau = DL @ self.opacity(f, i0, i1)
        ring = (A[:, None, :] @ -torch.expm1(-tau))[:, 0]
        return (rp ** 2 + ring) / self.spec.r_s ** 2

    def emission(self, f, i0, i1):
        """Planet-star flux ratio [b][i1 - i0]."""
        x, w = np.polynomial.legendre.leggauss(self.c["angles"])
        x, w = 0.5 * (x + 1.0), 0.5 * w
        K = self.opacity(f, i0, i1)
        dtau = K * (f["z"][:, 1:] - f["z"][:, :-1])[..., None] * f["inside"][..., None]
        below = torch.flip(torch.cumsum(torch.flip(dtau, [1]), 1), [1])       # tau at the bottom
        above = below - dtau
        nu = self.wn[i0:i1] * HC_K
        src = 1.0 / torch.expm1(nu / f["T"][..., None])
        surf = 1.0 / torch.expm1(nu / f["t_surf"])
        star = 1.0 / torch.expm1(nu / T_STAR)
        flux = 0.0
        for xk, wk in zip(x, w):
            part = torch.exp(-above / xk) * -torch.expm1(-dtau / xk)
            flux = flux + xk * wk * ((src * part).sum(1) + surf * torch.exp(-below[:, 0] / xk))
        return flux / (star * float((x * w).sum())) * (f["rp"] / self.spec.r_s) ** 2

    def blocks(self, i0, i1, cells):
        """(items, columns) blocks of at most `cells` (item, layer, wavenumber) values."""
        n, N = self.c["items"], self.c["layers"]
        cols = max(1, min(i1 - i0, cells // N))
        step = max(1, cells // (N * cols))
        for b in range(0, n, step):
            yield slice(b, min(n, b + step)), [(w, min(i1, w + cols)) for w in range(i0, i1, cols)]

    def spectra(self, i0, i1):
        of = self.emission if self.c["kind"] == "emission" else self.depth
        rows = []
        with torch.no_grad():
            for b, cols in self.blocks(i0, i1, 40_000_000):
                f = self.profile(self.d(self.th[b]), self.nl[b])
                rows.append(torch.cat([of(f, *c) for c in cols], dim=1))
        return torch.cat(rows)

    def pullback(self, g, i0, i1):
        """sum_i g[b][i] dD[b][i0 + i] / dtheta[b]."""
        out = []
        for b, cols in self.blocks(i0, i1, 6_000_000):
            th = self.d(self.th[b]).requires_grad_(True)
            total = torch.zeros_like(th)
            for c in cols:
                f = self.profile(th, self.nl[b])
                total += torch.autograd.grad((self.depth(f, *c) * g[b, c[0] - i0:c[1] - i0]).sum(), th)[0]
            out.append(total)
        return torch.cat(out)


def exact(case, seed):
    c = case
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    w, i0, i1 = _bin_matrix(c, dev)
    wsum = w.sum(0)
    if c["kind"] == "instrument":
        flux, sigma, z = _instrument_inputs(c, seed, i1 - i0, dev)
        binned = flux @ w / wsum
        noise = (binned.amax(1, keepdim=True) / SNR / math.sqrt(N_OBS)).expand_as(binned)
        return {"binned": binned, "binned_sigma": torch.sqrt(sigma ** 2 @ w ** 2) / wsum,
                "obs": binned + noise * z, "noise": noise.contiguous()}
    m = _Model(c, seed)
    if c["kind"] in ("model", "graph", "spectra", "emission"):
        native = m.spectra(0, c["wavenumbers"])
        binned = native[:, i0:i1] @ w / wsum
        if c["kind"] == "model":
            return {"native": native[0], "binned": binned[0]}
        return {"native": native, "binned": binned, "status": None}
    binned = m.spectra(i0, i1) @ w / wsum
    if c["kind"] == "binned":
        return {"binned": binned, "status": None}
    if c["kind"] == "gradient":
        r = (binned - m.d(m.obs)) / m.d(m.sig)
        grad = m.pullback((2.0 * r / m.d(m.sig) / wsum) @ w.T, i0, i1)
        return {"chi2": (r ** 2).sum(1), "grad": grad, "binned": binned, "status": None}
    rows = []
    for j in range(c["bins"]):
        at = torch.nonzero(w[:, j])[:, 0]
        a, b = int(at[0]), int(at[-1]) + 1
        rows.append(m.pullback((w[a:b, j] / wsum[j]).expand(c["items"], -1), i0 + a, i0 + b))
    return {"binned": binned, "jac": torch.stack(rows, dim=1), "status": None}
