"""The FP64 flux kernel's own Riemann finish (float start, one FP64 step),
limiter and divisions where they can go wrong, against the oracle at the FP64
tolerance of the parity tests (1e-12 of a particle's summed |flux|): adiabatic
indices with and without integer exponents, pressure ratios over many decades,
supersonic approach and recession (vacuum), and units whose pressures lie
outside the float range the start works in."""
import numpy as np
import pytest

from parity_util import compare, gpu_stages, oracle_stages

pytestmark = pytest.mark.gpu


def _state(wl, gamma, spread, mach, unit, seed):
    w = wl.lattice_wave(9, seed=seed, gamma=gamma, jitter=0.08)
    rng = np.random.default_rng(seed)
    n = w["x"].size
    m = w["m"] * np.exp(0.5 * rng.standard_normal(n))
    p = unit * np.exp(spread * rng.standard_normal(n))
    cs = np.sqrt(gamma * p * 9.0 ** -3 / m)
    v = rng.standard_normal((3, n)) * mach * cs
    U = p * 9.0 ** -3 / (gamma - 1.0)
    w.update(m=m, px=m * v[0], py=m * v[1], pz=m * v[2], U=U, E=U + 0.5 * m * (v * v).sum(0))
    return w


STATES = [
    # gamma, spread of ln p, Mach number, unit of the pressure
    (5.0 / 3.0, 0.3, 0.1, 1.0),      # near-equal states (most faces of a smooth flow)
    (5.0 / 3.0, 3.0, 2.0, 1.0),      # strong shocks and fans
    (5.0 / 3.0, 1.0, 8.0, 1.0),      # supersonic: pre-shock states, vacuum
    (1.4, 2.0, 1.0, 1.0),
    (2.0, 2.0, 1.0, 1.0),
    (1.3, 2.0, 1.0, 1.0),            # no integer exponent: pow()
    (1.05, 1.0, 0.5, 1.0),
    (5.0 / 3.0, 2.0, 1.0, 1e-34),    # float start out of range: the plain iteration
    (5.0 / 3.0, 2.0, 1.0, 1e34),
]
# (HLLC under MFV only where its outer waves do not overlap: where both point
# across the face, its flux depends on which of the two particles is called
# left, and the library and the oracle name them by different rules)
CASES = [(r, s, c) for c in STATES for r in ("exact", "hllc") for s in ("mfv", "mfm")
         if not (r == "hllc" and s == "mfv" and c[2] > 0.5)]


@pytest.mark.parametrize("riemann,scheme,state", CASES)
def test_fp64_fluxes_match_oracle(orc, riemann, scheme, state):
    gamma, spread, mach, unit = state
    from paper_2211_12243_gb300 import hydro, workloads
    w = _state(workloads, gamma, spread, mach, unit, 3)
    opts = dict(scheme=scheme, riemann=riemann)
    dt = 1e-3 / np.sqrt(unit)
    o = oracle_stages(orc, orc.config(gamma=gamma, **opts), w, dt)
    H = hydro.Hydro(hydro.default_config(gamma=gamma, precision="fp64", **opts))
    g = gpu_stages(hydro, H, w, dt)
    errs, bad = compare(g, o, 1e-12, what=("h", "omega", "B", "grad", "ncond", "dQ"))
    assert not bad, errs


@pytest.mark.parametrize("scheme", ["mfv", "mfm"])
def test_fp64_flux_sums_repeat(scheme):
    """The sums of the faces' contributions, whose additions arrive in any order:
    the rounding errors are summed beside them, so repeated calls agree to the
    rounding of the total (one unit in its last place) and of the errors' sum
    (2^-53 of at most 200 errors of 2^-53 of the largest contribution)."""
    import torch
    from paper_2211_12243_gb300 import hydro, workloads
    w = workloads.lognormal(30011, seed=4, grid=32, contrast=100.0)
    H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], scheme=scheme))
    H.set_boxes(*hydro.single_box(w))
    st = hydro.to_device(w)
    assert H.step(st, 1e-9, check=False)["status"] in (0, -5)   # (smoothing lengths)
    H.build_neighbours(st, st["h"] * 1.05, export=False)
    H.density(st)
    B, G, A, _ = H.gradients(st)
    dQ = np.stack([H.fluxes(st, B, G, A, 1e-3).cpu().numpy()[:, :5] for _ in range(8)])
    spread = dQ.max(0) - dQ.min(0)
    bound = np.spacing(np.abs(dQ).max(0)) + 200 * 2.0 ** -106 * np.abs(dQ).max((0, 1))
    assert np.all(spread <= bound)
    H.close()
