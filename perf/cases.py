"""The performance cases of the library: what is timed, on which inputs, and what it computes.

Each case is work that a user of the package has it do through `paper_2507_11603_gb300.thor`:
photon runs through gridless shells (homologous and power-law, H I and Mg II), photon runs
through Cartesian grids with peeling-off, the served stream of shell models, the reweighting
of a sweep's photon records, and forest optical depths.  Sizes are those of the benchmark's
workloads and of the tests, or parts of them that finish within about a second.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  what a program has in hand before the call
  run(state)           one pass through the public entry points
  work(case)           bytes and operations that a pass cannot do without
  exact(case, seed)    the outputs in 64 bits, where they have such a value

A Monte Carlo run's outputs are counts, fixed by the seed and the photon ids; images are
FP32 sums in no fixed order.  `exact` covers the deterministic sums (forest, reweighting).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_11603_gb300 import synth, thor

_PC = synth.PC_CM
_EW3 = 3.0 / 1215.67 * 299792.458  # equivalent width of 3 Angstrom in km/s
_COUNTS = ("n_escaped", "n_absorbed", "n_capped", "n_scat", "n_dust_scat", "n_upar_iters", "n_steps")
_ctx = None


def _context():
    """One context per process, as a program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = thor.Context(0)
    return _ctx


def listed():
    return [
        # The smallest call: a few hundred photons through a thin static sphere, host buffers
        # (a quick look, a unit of a parameter scan): launches, copies and synchronisation.
        {"name": "shell_tiny", "kind": "shell", "n_photons": 256, "tau0": 10.0, "N_HI": 0.0, "T": 1e4, "R_in": 0.0,
         "v_max": 0.0, "tau_dust": 0.0, "phase": "isotropic", "core_skip": False, "sigma": 0.0, "n_bins": 200,
         "X_lim": 500.0, "device": False, "raw": False, "max_scat": 0},
        # The static sphere that validation runs use: tau0 = 1e4, 5000 photons at line centre.
        {"name": "sphere_1e4", "kind": "shell", "n_photons": 5000, "tau0": 1e4, "N_HI": 0.0, "T": 1e4, "R_in": 0.0,
         "v_max": 0.0, "tau_dust": 0.0, "phase": "isotropic", "core_skip": False, "sigma": 0.0, "n_bins": 200,
         "X_lim": 513.8, "device": False, "raw": False, "max_scat": 0},
        # The expanding dusty shell of the benchmark at a tenth of its column, so that a pass
        # takes under a second: 1e5 photons to completion, records per photon, device buffers.
        {"name": "shell_outflow", "kind": "shell", "n_photons": 100000, "tau0": 0.0, "N_HI": 1e19, "T": 1e4,
         "R_in": 0.9, "v_max": 200.0, "tau_dust": 0.5, "phase": "dipole", "core_skip": False, "sigma": 50.0,
         "n_bins": 400, "X_lim": 1500.0, "device": True, "raw": True, "max_scat": 0},
        # The benchmark's full column with core-skipping, as the served models run it.
        {"name": "shell_core_skip", "kind": "shell", "n_photons": 20000, "tau0": 0.0, "N_HI": 1e20, "T": 1e4,
         "R_in": 0.9, "v_max": 200.0, "tau_dust": 0.5, "phase": "dipole", "core_skip": True, "sigma": 50.0,
         "n_bins": 400, "X_lim": 1500.0, "device": False, "raw": False, "max_scat": 0},
        # The transport run of a shell-model sweep: power-law shell, line on a continuum, the
        # records that the reweighting takes, on the device.
        {"name": "sweep_transport", "kind": "power_law", "species": "HI", "n_photons": 200000, "log_N": 18.4,
         "T": 1e4, "R_in": 0.1, "v_max": 120.0, "alpha_rho": -0.5, "alpha_v": 1.0, "tau_dust": 0.0, "X0": 0.0,
         "sigma": 800.0, "ew": _EW3, "C": 2500.0, "n_bins": 400, "X_lo": -2500.0, "X_hi": 2500.0},
        # The Mg II doublet through an outflowing sphere lit by a flat continuum.
        {"name": "mgii_sphere", "kind": "power_law", "species": "MgII", "n_photons": 100000, "log_N": 14.5, "T": 1e4,
         "R_in": 1e-3, "v_max": 100.0, "alpha_rho": 0.0, "alpha_v": 1.0, "tau_dust": 0.0, "X0": -400.0,
         "sigma": 100.0, "ew": 0.0, "C": 1400.0, "n_bins": 300, "X_lo": -2000.0, "X_hi": 1000.0},
        # The post-processing of that sweep: 2e5 photon records on the device reweighted to 256
        # intrinsic spectra and dust depths.
        {"name": "sweep_reweight", "kind": "reweight", "n": 200000, "n_targets": 256, "n_bins": 400, "device": True},
        # A burst of served shell models: 24 requests of the stream's parameter ranges at once.
        {"name": "served_burst", "kind": "served", "requests": 24, "nhi_max": 1e19, "core_skip": True},
        # The 256^3 grid with peeling-off to three observers, photons stopped at 1000
        # scatterings: the regime of a long run, with all packets in flight.
        {"name": "grid_peel_256", "kind": "grid", "nx": 256, "ny": 256, "nz": 256, "n_photons": 200000, "n_mean": 1e-3,
         "peel": True, "img_n": 128, "peel_bins": 256, "max_scat": 1000, "phase": "dipole", "new_grid": False},
        # A small ragged grid that comes with the call (fields on the host, thin gas, records per
        # photon instead of images): building the geometry is part of the work.
        {"name": "grid_small_new", "kind": "grid", "nx": 48, "ny": 40, "nz": 36, "n_photons": 20000, "n_mean": 1e-7,
         "peel": False, "img_n": 0, "peel_bins": 0, "max_scat": 0, "phase": "mixed", "new_grid": True},
        # Forest optical depths of a device-resident box at the full column length and bin count.
        {"name": "forest_box", "kind": "forest", "nz": 1024, "ny": 64, "nx": 64, "n_bins": 2048, "dv_cell": 2.0,
         "first": 0, "count": 4096, "device": True},
        # A few short skewers of odd sizes from host arrays.
        {"name": "forest_skewers", "kind": "forest", "nz": 300, "ny": 5, "nx": 7, "n_bins": 250, "dv_cell": 5.5,
         "first": 3, "count": 29, "device": False},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["shell", "shell", "power_law", "reweight", "served", "grid", "grid", "forest", "forest"])
    if kind == "shell":
        moving = rng.random() < 0.7
        return {"kind": "shell", "n_photons": int(_log(rng, 64, 60000)), "tau0": 0.0 if moving else _log(rng, 1.0, 3e4),
                "N_HI": _log(rng, 1e16, 6e18) if moving else 0.0, "T": _log(rng, 8e3, 1e5),
                "R_in": rng.choice([0.2, 0.5, 0.9]) if moving else 0.0, "v_max": rng.uniform(100.0, 500.0) if moving else 0.0,
                "tau_dust": rng.choice([0.0, 0.3, 1.0, 2.0]) if moving else 0.0,
                "phase": rng.choice(["isotropic", "dipole", "mixed"]), "core_skip": rng.random() < 0.4,
                "sigma": rng.choice([0.0, 20.0, 50.0]), "n_bins": rng.randrange(33, 700),
                "X_lim": 1500.0, "device": rng.random() < 0.5, "raw": rng.random() < 0.5,
                "max_scat": rng.choice([0, 0, 5000])}
    if kind == "power_law":
        mg = rng.random() < 0.4
        return {"kind": "power_law", "species": "MgII" if mg else "HI", "n_photons": int(_log(rng, 1000, 200000)),
                "log_N": rng.uniform(13.0, 14.6) if mg else rng.uniform(16.5, 18.4), "T": _log(rng, 1e4, 5e4),
                "R_in": 1e-3 if mg else rng.choice([0.1, 0.2, 0.5]), "v_max": rng.uniform(80.0, 300.0),
                "alpha_rho": 0.0 if mg else rng.uniform(-1.5, 0.0), "alpha_v": 1.0 if mg else rng.uniform(0.5, 1.2),
                "tau_dust": 0.0 if mg else rng.choice([0.0, 0.4]), "X0": -400.0 if mg else 0.0,
                "sigma": 100.0 if mg else 800.0, "ew": 0.0 if mg else _EW3, "C": 1400.0 if mg else 2500.0,
                "n_bins": rng.randrange(50, 500), "X_lo": -2500.0, "X_hi": 2500.0}
    if kind == "reweight":
        return {"kind": "reweight", "n": int(_log(rng, 5000, 200000)), "n_targets": int(_log(rng, 1, 256)),
                "n_bins": rng.randrange(50, 500), "device": rng.random() < 0.7}
    if kind == "served":
        return {"kind": "served", "requests": rng.randrange(2, 20), "nhi_max": _log(rng, 2e17, 5e18),
                "core_skip": rng.random() < 0.7}
    if kind == "grid":
        if rng.random() < 0.5:
            return {"kind": "grid", "nx": rng.randrange(8, 80), "ny": rng.randrange(8, 80), "nz": rng.randrange(8, 80),
                    "n_photons": int(_log(rng, 300, 30000)), "n_mean": _log(rng, 1e-9, 1e-7), "peel": False, "img_n": 0,
                    "peel_bins": 0, "max_scat": 0, "phase": rng.choice(["dipole", "mixed", "isotropic"]),
                    "new_grid": rng.random() < 0.5}
        img = rng.choice([16, 32])
        return {"kind": "grid", "nx": img * rng.randrange(1, 8), "ny": img * rng.randrange(1, 8),
                "nz": img * rng.randrange(1, 8), "n_photons": int(_log(rng, 1000, 150000)), "n_mean": _log(rng, 1e-6, 1e-3),
                "peel": True, "img_n": img, "peel_bins": rng.randrange(40, 257), "max_scat": rng.randrange(100, 1001),
                "phase": rng.choice(["dipole", "mixed", "isotropic"]), "new_grid": False}
    nz = int(_log(rng, 60, 1500))
    nx, ny = rng.randrange(1, 49), rng.randrange(1, 49)
    first = rng.randrange(0, max(1, nx * ny // 4))
    return {"kind": "forest", "nz": nz, "ny": ny, "nx": nx, "n_bins": rng.randrange(40, 2049), "dv_cell": rng.uniform(1.0, 8.0),
            "first": first, "count": rng.randrange(1, nx * ny - first + 1), "device": rng.random() < 0.6}


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _field(shape, sigma, g):
    """A Gaussian random field with P(k) ~ k^-11/3 scaled to `sigma`, as the synthetic inputs have it."""
    f = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda"))
    k = [torch.fft.fftfreq(n, device="cuda") for n in shape[:-1]] + [torch.fft.rfftfreq(shape[-1], device="cuda")]
    k2 = sum(ki.pow(2).reshape([-1 if j == i else 1 for j in range(3)]) for i, ki in enumerate(k))
    f = torch.where(k2 > 0, f * k2.clamp_min(1e-30).pow(-11.0 / 12.0), torch.zeros_like(f))
    v = torch.fft.irfftn(f, s=shape)
    v = v - v.mean()
    s = v.std() if v.numel() > 1 else v.new_zeros(())
    return (v * (sigma / s if float(s) > 0 else 0.0)).float().contiguous()


def _grid_fields(c, seed):
    g = _gen(seed)
    shape = (c["nz"], c["ny"], c["nx"])
    n = c["n_mean"] * torch.exp(1.5 * torch.randn(shape, generator=g, device="cuda") - 0.5 * 1.5 ** 2)
    T = 1e4 * torch.exp(0.5 * torch.randn(shape, generator=g, device="cuda"))
    v = torch.stack([_field(shape, 50.0, g) for _ in range(3)])
    kd = (0.01 * 4e-22) * n
    f = [n.float().contiguous(), T.float().contiguous(), v.contiguous(), kd.float().contiguous()]
    return [x.cpu().numpy() for x in f] if c["new_grid"] else f


def _forest_fields(c, seed):
    g = _gen(seed)
    shape = (c["nz"], c["ny"], c["nx"])
    ratio = torch.exp(2.0 * torch.randn(shape, generator=g, device="cuda") - 2.0)
    f = [(1e-10 * ratio).float().contiguous(), (1e4 * ratio.pow(0.6)).float().contiguous(), _field(shape, 30.0, g)]
    return f if c["device"] else [x.cpu().numpy() for x in f]


def _records(c, seed):
    """Photon records as a sweep's transport run leaves them: emitted and escaping frequencies,
    columns, most photons escaped; and targets over the sweep's ranges."""
    g = _gen(seed)
    n = c["n"]
    line = torch.rand(n, generator=g, device="cuda") < _EW3 / (_EW3 + 5000.0)
    X0 = torch.where(line, 800.0 * torch.randn(n, generator=g, device="cuda"),
                     2500.0 * (2.0 * torch.rand(n, generator=g, device="cuda") - 1.0))
    X = X0 + 300.0 * torch.randn(n, generator=g, device="cuda")
    col = torch.exp(0.7 * torch.randn(n, generator=g, device="cuda"))
    st = torch.where(torch.rand(n, generator=g, device="cuda") < 0.9, 1, 2).to(torch.uint8)
    rng = np.random.default_rng(seed)
    K = c["n_targets"]
    targets = np.stack([rng.uniform(100.0, 800.0, K), rng.uniform(10.0, 200.0, K) / 1215.67 * 299792.458,
                        np.full(K, 2500.0), rng.uniform(0.0, 2.0, K)], axis=1)
    r = [X0.float(), X.float(), col.float(), st]
    return (r if c["device"] else [x.cpu().numpy() for x in r]), targets


def _grid(ctx, c, f):
    return ctx.grid(*f, 100 * _PC, phase=c["phase"])


def prepare(case, seed):
    c, ctx = dict(case), _context()
    s = {"case": c, "seed": seed}
    if c["kind"] == "shell":
        s["geom"] = ctx.shell(T=c["T"], R_in=c["R_in"], N_HI=c["N_HI"], tau0=c["tau0"], v_max=c["v_max"],
                              tau_dust=c["tau_dust"], phase=c["phase"], core_skip=c["core_skip"])
    elif c["kind"] == "power_law":
        s["geom"] = ctx.shell(profile="power_law", species=c["species"], T=c["T"], R_in=c["R_in"],
                              N_HI=10.0 ** c["log_N"], v_max=c["v_max"], alpha_rho=c["alpha_rho"],
                              alpha_v=c["alpha_v"], tau_dust=c["tau_dust"], phase="dipole")
    elif c["kind"] == "grid":
        s["fields"] = _grid_fields(c, seed)
        if not c["new_grid"]:
            s["geom"] = _grid(ctx, c, s["fields"])
            del s["fields"]
    elif c["kind"] == "forest":
        s["fields"] = _forest_fields(c, seed)
    elif c["kind"] == "reweight":
        s["records"], s["targets"] = _records(c, seed)
    else:
        s["server"] = ctx.server(max_requests=64)
        s["models"] = synth.shell_stream(c["requests"], seed=seed, nhi_max=c["nhi_max"])
    return s


# ------------------------------------------------------------------------------ passes
def _out(r):
    d = {"spectrum": r.spectrum, "ends": [r.underflow, r.overflow], "counts": [r.stats[k] for k in _COUNTS]}
    for k in ("cube", "raw_X", "raw_nscat", "raw_status", "raw_X0", "raw_col"):
        if getattr(r, k) is not None:
            d[k] = getattr(r, k)
    return d


def run(state):
    c, ctx = state["case"], _context()
    if c["kind"] == "shell":
        return _out(ctx.run(state["geom"], n_photons=c["n_photons"], seed=state["seed"], sigma=c["sigma"],
                            n_bins=c["n_bins"], X_min=-c["X_lim"], X_max=c["X_lim"], raw=c["raw"],
                            max_scat=c["max_scat"], device_out=c["device"]))
    if c["kind"] == "power_law":
        return _out(ctx.run(state["geom"], n_photons=c["n_photons"], seed=state["seed"], X0=c["X0"], sigma=c["sigma"],
                            ew=c["ew"], C_cont=c["C"], n_bins=c["n_bins"], X_min=c["X_lo"], X_max=c["X_hi"], raw=True,
                            raw_sweep=True, device_out=True))
    if c["kind"] == "grid":
        g = _grid(ctx, c, state["fields"]) if c["new_grid"] else state["geom"]
        kw = dict(peel=True, img_n=c["img_n"], peel_bins=c["peel_bins"], device_out=True) if c["peel"] else dict(raw=True)
        r = ctx.run(g, n_photons=c["n_photons"], seed=state["seed"], n_bins=256, X_min=-1000.0, X_max=1000.0,
                    max_scat=c["max_scat"], **kw)
        if c["new_grid"]:
            g.close()
        return _out(r)
    if c["kind"] == "forest":
        return ctx.forest(*state["fields"], ds_cm=synth.forest_scale(2.0, c["dv_cell"]), dv_cell=c["dv_cell"],
                          n_bins=c["n_bins"], dv_bin=c["nz"] * c["dv_cell"] / c["n_bins"], first=c["first"],
                          count=c["count"])
    if c["kind"] == "reweight":
        return ctx.reweight(*state["records"], sample=(800.0, _EW3, 2500.0), targets=state["targets"],
                            n_bins=c["n_bins"], X_min=-2500.0, X_max=2500.0)
    srv = state["server"]
    tickets = [srv.submit(N_HI=m["N_HI"], T=m["T"], v_max=m["v_max"], tau_dust=m["tau_dust"], n_photons=m["n_photons"],
                          seed=m["seed"], R_in=0.9, phase="dipole", sigma=50.0, core_skip=c["core_skip"])
               for m in state["models"]]
    rs = [srv.wait(t, timeout_ms=600000) for t in tickets]
    return {"spectra": np.stack([r.spectrum for r in rs]), "ends": [[r.underflow, r.overflow] for r in rs][:4],
            "counts": np.array([[r.stats[k] for k in _COUNTS] for r in rs], dtype=np.int64)}


# ------------------------------------------------------------------------------ work
def _sigma0(vth_cms):
    """Line-centre cross-section [cm^2] of Lyman alpha: f12 sqrt(pi) e^2 lambda0 / (m_e c v_th)."""
    return 0.4164 * math.sqrt(math.pi) * 4.80320471e-10 ** 2 * 1215.67e-8 / (9.1093837015e-28 * 2.99792458e10 * vth_cms)


_EVENT = 400.0  # operations of one photon event: random words, Voigt profile, velocities, direction


def _events(c):
    """Scatterings per photon, about (n_scat of the runs, fitted): what the histories cannot do without."""
    if c["kind"] == "shell":
        tau0 = c["tau0"] or c["N_HI"] * _sigma0(12845.07 * math.sqrt(c["T"]))
        per = 1.0 + (0.9 * tau0 if c["v_max"] == 0.0 else 0.01 * tau0)
        return min(per, c["max_scat"]) if c["max_scat"] else per
    if c["kind"] == "power_law":
        return 3.0 if c["species"] == "MgII" else 2e-16 * 10.0 ** c["log_N"]
    if c["kind"] == "grid":
        return float(c["max_scat"]) if c["n_mean"] > 1e-5 and c["max_scat"] else 30.0
    return 1e3 * c["nhi_max"] / 1e19


def work(case):
    c = dict(case)
    if c["kind"] == "forest":
        used = c["count"] * c["nz"]
        return {"bytes": 12 * used + 4 * c["count"] * c["n_bins"], "flops": 22 * used * c["n_bins"]}
    if c["kind"] == "reweight":
        return {"bytes": 13 * c["n"] + 40 * c["n_targets"] + 8 * c["n_targets"] * (c["n_bins"] + 2),
                "flops": 30 * c["n"] * c["n_targets"]}
    n = c["requests"] * 20000 if c["kind"] == "served" else c["n_photons"]
    b = 8 * (c.get("n_bins", 400) + 2)
    if c["kind"] == "grid":
        cells = c["nx"] * c["ny"] * c["nz"]
        b += 24 * cells if c["new_grid"] else 32 * min(cells, c["n_photons"])
        b += 12 * c["img_n"] ** 2 * c["peel_bins"] + (0 if c["peel"] else 9 * n)
    elif c["kind"] == "power_law" or c.get("raw"):
        b += (17 if c["kind"] == "power_law" else 9) * n
    return {"bytes": b, "flops": _EVENT * n * (1.0 + _events(c))}


# ------------------------------------------------------------------------------ 64 bits
def _voigt64(a, x):
    """H(a, x) = (a / pi) int e^{-t^2} / ((x - t)^2 + a^2) dt by the trapezoidal rule with step
    h = 1/2 and the residue of the pole it passes over (Hunter and Regan 1972), in 64 bits."""
    h = 0.5
    s = torch.zeros_like(x)
    a2 = a * a
    for n in range(-13, 13):
        t = (n + 0.5) * h  # nodes at odd multiples of h / 2
        s += math.exp(-t * t) / ((x - t) ** 2 + a2)
    s *= h * a / math.pi
    # residue: Re[2 e^{-z^2} / (1 + e^{-2 pi i z / h})] with z = x + i a, for these nodes
    near = (x.abs() < 7.5).nonzero(as_tuple=True)
    z = torch.complex(x[near], a.expand_as(x)[near])
    s[near] += (2.0 * torch.exp(-z * z) / (1.0 + torch.exp(-2j * math.pi / h * z))).real
    return s


def _forest64(c, seed):
    n, T, v = (x.double() if torch.is_tensor(x) else torch.from_numpy(x).cuda().double() for x in _forest_fields(c, seed))
    cols = torch.arange(c["first"], c["first"] + c["count"], device="cuda")
    n, T, v = (x.reshape(c["nz"], -1)[:, cols].T.contiguous() for x in (n, T, v))
    V, db = c["nz"] * c["dv_cell"], c["nz"] * c["dv_cell"] / c["n_bins"]
    vth = 1e-5 * torch.sqrt(2.0 * 1.380649e-16 * T / 1.6735575e-24)  # km/s
    a = 6.265e8 * 1215.67e-8 / (4.0 * math.pi * 1e5 * vth)
    amp = n * _sigma0(1e5 * vth) * synth.forest_scale(2.0, c["dv_cell"])
    vk = (torch.arange(c["nz"], device="cuda", dtype=torch.float64) + 0.5) * c["dv_cell"] + v
    vb = (torch.arange(c["n_bins"], device="cuda", dtype=torch.float64) + 0.5) * db
    out = torch.empty((c["count"], c["n_bins"]), dtype=torch.float64, device="cuda")
    rows = max(1, int(2e8 // (c["nz"] * c["n_bins"])))
    for i in range(0, c["count"], rows):
        j = slice(i, i + rows)
        d = vb[None, None, :] - vk[j, :, None]
        d = d - V * torch.round(d / V)
        H = _voigt64(a[j, :, None], d / vth[j, :, None])
        out[j] = torch.einsum("rk,rkb->rb", amp[j], H)
    return out if c["device"] else out.cpu().numpy()


def _reweight64(c, seed):
    (X0, X, col, st), targets = _records(c, seed)
    X0, X, col = (x.double() if torch.is_tensor(x) else torch.from_numpy(x).cuda().double() for x in (X0, X, col))
    st = st if torch.is_tensor(st) else torch.from_numpy(st).cuda()
    nb = c["n_bins"]
    # the bin of a photon is a whole number: single precision, as the records are
    f = (X.float() - (-2500.0)) * float(np.float32(nb / 5000.0))
    b = torch.where(f >= 0, torch.where(f >= nb, nb + 1, f.long()), nb)

    def pdf(sigma, ew, C):
        pl = ew / (ew + 2 * C)
        g = pl / (math.sqrt(2 * math.pi) * sigma) * torch.exp(-0.5 * (X0 / sigma) ** 2)
        return torch.where(X0.abs() <= C, g + (1 - pl) / (2 * C), g)

    ps, ok = pdf(800.0, _EW3, 2500.0), st == 1
    out = np.zeros((len(targets), nb + 2))
    for t, (sigma, ew, C, tau_d) in enumerate(targets):
        w = torch.where(ok, pdf(sigma, ew, C) / ps * torch.exp(-tau_d * col), torch.zeros_like(ps))
        out[t] = torch.zeros(nb + 2, dtype=torch.float64, device="cuda").index_add_(0, b, w).cpu().numpy() / c["n"]
    return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "forest" and c["count"] * c["nz"] * c["n_bins"] <= 10 ** 10:
        return _forest64(c, seed)
    if c["kind"] == "reweight":
        return _reweight64(c, seed)
    return None
