"""States at the edges of what a step accepts: positions of minus zero, cold
gas whose velocities are zeros of either sign, negative pressures, values that
are not numbers in the staged calls, densities beyond the float range, and
limiter factors that switch a bound off."""
import numpy as np
import pytest

from paper_2211_12243_gb300 import workloads as W
from parity_util import compare, gpu_stages, oracle_stages

pytestmark = pytest.mark.gpu


def _step(hydro, w, dt, **opts):
    import torch
    H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], **opts))
    H.set_boxes(*hydro.single_box(w))
    st = hydro.to_device(w)
    s = H.step(st, dt, check=False)
    torch.cuda.synchronize()
    out = {k: v.cpu().numpy() for k, v in st.items()}
    H.close()
    return s, out


def _cold(n, seed):
    """a jittered lattice without pressure or motion"""
    w = dict(W.lattice_wave(n, jitter=0.05, seed=seed))
    z = np.zeros(w["x"].size)
    w.update(m=np.full(z.size, 1.0 / z.size), px=z, py=z.copy(), pz=z.copy(), E=z.copy(), U=z.copy())
    return w


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_position_of_minus_zero_stays_in_the_box(precision):
    """x = -0.0 and a displacement that underflows to -0.0"""
    from paper_2211_12243_gb300 import hydro
    w = _cold(8, 1)
    w["x"][:5] = -0.0
    w["px"][:] = -1e-320
    s, out = _step(hydro, w, 1e-8, precision=precision)
    assert s["status"] in (0, -5), s
    assert np.all(out["x"][:5] == 0.0)
    assert np.all(out["x"] >= 0.0) and np.all(out["x"] < w["L"][0])


@pytest.mark.parametrize("scheme", ["mfv", "mfm"])
def test_cold_gas_with_zeros_of_either_sign(scheme):
    """no pressure, velocities +0 and -0: every face is a vacuum"""
    from paper_2211_12243_gb300 import hydro
    w = _cold(10, 2)
    rng = np.random.default_rng(3)
    for k in ("px", "py", "pz"):
        w[k] = np.copysign(0.0, rng.standard_normal(w["x"].size))
    s, out = _step(hydro, w, 1e-3, scheme=scheme)
    assert s["status"] in (0, -5), s
    assert s["vacuum_faces"] == s["flux_pairs"] > 0
    for k in ("m", "px", "E", "x", "y", "z"):
        assert np.array_equal(out[k], w[k]), k


@pytest.mark.parametrize("riemann,scheme", [("exact", "mfv"), ("exact", "mfm"), ("hllc", "mfm")])
def test_negative_pressure_is_reported(riemann, scheme):
    """a particle of negative internal energy: HYDRO_ENONFINITE, as the
    solver's square roots of negative numbers give"""
    from paper_2211_12243_gb300 import hydro
    w = dict(W.lattice_wave(10, jitter=0.05))
    for k in ("E", "U"):
        w[k] = w[k].copy()
        w[k][123] *= -0.1
    s, _ = _step(hydro, w, 1e-3, scheme=scheme, riemann=riemann)
    assert s["status"] == -7, s


@pytest.mark.parametrize("riemann,scheme", [("exact", "mfv"), ("exact", "mfm"), ("hllc", "mfv"),
                                            ("hllc", "mfm")])
def test_nan_gradients_reach_the_fluxes(riemann, scheme):
    """a velocity gradient that is not a number: the fluxes of that particle
    are not numbers either (they are not dropped as a vacuum's)"""
    import torch
    from paper_2211_12243_gb300 import hydro
    w = W.lattice_wave(9, jitter=0.05)
    H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], scheme=scheme, riemann=riemann,
                                         limiter=0, time_extrap=0))
    H.set_boxes(*hydro.single_box(w))
    st = hydro.to_device(w)
    H.build_neighbours(st, st["h"] * 1.3, export=False)
    H.density(st)
    B, G, A, N = H.gradients(st)
    G[77, 1, 0] = float("nan")
    dQ = H.fluxes(st, B, G, A, 1e-3)
    torch.cuda.synchronize()
    bad = ~np.isfinite(dQ.cpu().numpy()[:, :5])
    assert bad[77, 4] and np.count_nonzero(bad.any(1)) > 5
    H.close()


@pytest.mark.parametrize("scheme", ["mfv", "mfm"])
@pytest.mark.parametrize("unit", [1e-60, 1e-42, 1e42, 1e60])
def test_uniform_pressure_at_densities_beyond_float(orc, scheme, unit):
    from paper_2211_12243_gb300 import hydro
    w = dict(W.lattice_wave(9, jitter=0.08))
    n = w["x"].size
    rng = np.random.default_rng(5)
    w["m"] = unit / n * np.exp(0.3 * rng.standard_normal(n))
    dt = 1e-3 * np.sqrt(unit)
    # (the pressure the solver sees is U (gamma - 1) / omega: uniform to rounding)
    cfg = orc.config(gamma=w["gamma"], scheme=scheme, limiter=1)
    h, om, _, st = orc.density(cfg, w["x"], w["y"], w["z"], w["L"], w["h"])
    w["U"] = om / (w["gamma"] - 1.0)
    w["E"] = w["U"].copy()
    o = oracle_stages(orc, cfg, w, dt)
    H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], scheme=scheme))
    g = gpu_stages(hydro, H, w, dt)
    errs, bad = compare(g, o, 1e-12, what=("h", "omega", "B", "grad", "ncond", "dQ"))
    assert not bad, errs
    H.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["psi1", "psi2"])
def test_infinite_limiter_factors(precision, name):
    """a factor beyond the float range switches its bound off, also where the
    two cells are equal (a fluid at rest)"""
    from paper_2211_12243_gb300 import hydro
    w = W.sod(8)
    ref, a = _step(hydro, w, 1e-3, precision=precision, **{name: 1e30})
    s, b = _step(hydro, w, 1e-3, precision=precision, **{name: float("inf")})
    assert s["status"] == ref["status"] == 0, s
    for k in ("m", "px", "py", "pz", "E"):
        assert np.max(np.abs(a[k] - b[k])) <= 1e-6 * np.max(np.abs(a[k])), k


@pytest.mark.parametrize("gap", [1e-156, 1e-161])
def test_particles_whose_squared_distance_is_subnormal(orc, gap):
    """two pairs of particles closer than 1e-154: as coincident ones, not NaN"""
    from paper_2211_12243_gb300 import hydro
    w = dict(W.lattice_wave(9, jitter=0.08))
    for k in ("x", "y", "z"):
        w[k] = w[k].copy()
        w[k][100:102] = 0.0
        w[k][300:302] = 0.0
    w["x"][101] = gap
    w["y"][300:302] = 0.5
    w["z"][301] = gap
    opts = dict(n_ngb=48.0)
    o = oracle_stages(orc, orc.config(gamma=w["gamma"], **opts), w, 1e-3)
    H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], **opts))
    g = gpu_stages(hydro, H, w, 1e-3, search=1.6)
    errs, bad = compare(g, o, 1e-12, what=("h", "omega", "B", "grad", "ncond", "dQ"))
    assert not bad, errs
    H.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_smoothing_length_that_is_not_a_number(precision):
    """staged calls with one such h: that particle has no pairs, so its matrix is
    singular (B and gradient 0) and its faces carry nothing; particles out of its
    reach keep their values"""
    import torch
    from paper_2211_12243_gb300 import hydro
    w = W.lattice_wave(12, jitter=0.05)
    H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], precision=precision))
    H.set_boxes(*hydro.single_box(w))
    st = hydro.to_device(w)
    H.build_neighbours(st, st["h"] * 1.3, export=False)
    H.density(st)
    ref = H.gradients(st)
    dQ0 = H.fluxes(st, *ref[:3], 1e-3)
    st["h"][100] = float("nan")
    B, G, A, N = H.gradients(st)
    assert torch.all(B[100] == 0) and torch.all(G[100] == 0) and torch.isinf(N[100])
    other = torch.arange(B.shape[0], device="cuda") != 100
    for a, b in zip(ref, (B, G, A, N)):
        assert torch.equal(a[other], b[other])
    dQ = H.fluxes(st, *ref[:3], 1e-3)
    assert torch.all(dQ[100] == 0) and torch.isfinite(dQ).all()
    same = (dQ - dQ0).abs().amax(1) <= 1e-12 * dQ0.abs().max()
    assert int((~same).sum()) < 120       # (its neighbours)
    H.close()
