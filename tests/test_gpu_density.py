"""Smoothing lengths where the density kernels branch, against the oracle
(1e-12 relative in FP64, as the parity tests): separations too small against
the box for the float iteration, both kernels and large N_NGB, and guard
rounds whose re-solves walk lists longer than a warp's cache."""
import numpy as np
import pytest

from paper_2211_12243_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hyd():
    from paper_2211_12243_gb300 import hydro
    return hydro


def _cluster(scale, n=3001, seed=1):
    """n particles in a ball of radius ~scale of the unit box"""
    rng = np.random.default_rng(seed)
    p = 0.37 + scale * rng.standard_normal((3, n))
    d = np.linalg.norm(p - 0.37, axis=0)
    return p, 0.7 * scale * np.exp(0.33 * (d / scale) ** 2) * n ** (-1.0 / 3.0) * 4.0


@pytest.mark.parametrize("precision,scale", [("fp64", 1e-2), ("fp64", 3e-5), ("fp64", 1e-7),
                                             ("fp64", 1e-9), ("mixed", 1e-2)])
@pytest.mark.parametrize("kernel,n_ngb", [("wendland", 32.0), ("cubic", 64.0)])
def test_density_of_a_small_cluster(orc, hyd, precision, scale, kernel, n_ngb):
    import torch
    (x, y, z), h0 = _cluster(scale)
    n, L = x.size, np.ones(3)
    co = orc.config(kernel=kernel, n_ngb=n_ngb)
    h, om, _, st = orc.density(co, x, y, z, L, h0)
    assert st == 0
    H = hyd.Hydro(hyd.default_config(precision=precision, kernel=kernel, n_ngb=n_ngb))
    H.set_boxes(np.array([0, n], dtype=np.int64), L)
    dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")
    s = {"x": dev(x), "y": dev(y), "z": dev(z), "h": dev(h0), "omega": dev(np.zeros(n))}
    H.build_neighbours(s, dev(h * 1.2), export=False)
    H.density(s)
    # (the mixed path's positions are 64-bit fixed point in the box: 5e-20 L)
    assert np.max(np.abs(s["h"].cpu().numpy() / h - 1)) < 1e-12
    assert np.max(np.abs(s["omega"].cpu().numpy() / om - 1)) < 4e-12
    H.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,n_ngb", [(5003, 32.0), (6007, 250.0)])
def test_guard_resolves_long_lists(orc, hyd, precision, n, n_ngb):
    rng = np.random.default_rng(5)
    w = W.lattice_wave(4)
    m = np.full(n, 1.0 / n)
    w = W._pack(rng.random(n), rng.random(n), rng.random(n), m, 0 * m, 0 * m, 0 * m,
                np.full(n, 1.5), W._h_guess(np.full(n, float(n)), n_ngb), (1.0, 1.0, 1.0),
                5.0 / 3.0, "random")
    kw = dict(n_ngb=n_ngb, ncond_crit=1.1 if n_ngb > 100 else 1.6)
    so, _, info = orc.step(orc.config(gamma=w["gamma"], **kw), w, 1e-4)
    H = hyd.Hydro(hyd.default_config(gamma=w["gamma"], precision=precision, **kw))
    H.set_boxes(*hyd.single_box(w))
    st = hyd.to_device(w)
    stats = H.step(st, 1e-4, check=False)
    assert stats["ngb_rounds"] >= 1 and stats["status"] in (0, -5)
    err = np.abs(st["h"].cpu().numpy() / so["h"] - 1)
    grown = so["h"] > 1.03 * np.median(so["h"])
    assert grown.any()
    if precision == "fp64":
        assert err.max() < 1e-12
    else:
        # a float E may put a particle on the other side of the threshold
        assert np.mean(err > 1e-12) < 2e-3
    H.close()


@pytest.mark.parametrize("n", [4099, 20011])
def test_density_where_the_float_iteration_does_not_settle(orc, hyd, n):
    """near-coincident pairs: the float sums jump by two at a time and the
    iteration may wander at its tolerance; FP64 converges from the guess"""
    import torch
    rng = np.random.default_rng(n)
    c = rng.random((3, n))
    c[:, n - n // 2:] = c[:, :n // 2] + 1e-8
    c = np.minimum(c, 1 - 1e-12)
    h0 = np.full(n, np.cbrt(24.0 / np.pi / n))
    h, om, _, st = orc.density(orc.config(), *c, np.ones(3), h0)
    assert st == 0
    H = hyd.Hydro(hyd.default_config())
    H.set_boxes(np.array([0, n], dtype=np.int64), np.ones(3))
    dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")
    s = {"x": dev(c[0]), "y": dev(c[1]), "z": dev(c[2]), "h": dev(h0), "omega": dev(np.zeros(n))}
    H.build_neighbours(s, dev(h * 1.2), export=False)
    H.density(s)
    assert np.max(np.abs(s["h"].cpu().numpy() / h - 1)) < 1e-12
    H.close()


@pytest.mark.parametrize("n", [131, 8192, 8193])
def test_warp_and_thread_solves_agree(orc, hyd, n):
    """either side of the size up to which a warp solves each particle"""
    import torch
    rng = np.random.default_rng(n)
    c = rng.random((3, n))
    n_ngb = 32.0 if n > 1000 else 18.0
    h0 = np.full(n, np.cbrt(3 * n_ngb / (4 * np.pi * max(n, 40))))
    h, om, _, st = orc.density(orc.config(n_ngb=n_ngb), *c, np.ones(3), h0)
    assert st == 0
    for precision in ("fp64", "mixed"):
        H = hyd.Hydro(hyd.default_config(precision=precision, n_ngb=n_ngb))
        H.set_boxes(np.array([0, n], dtype=np.int64), np.ones(3))
        dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")
        s = {"x": dev(c[0]), "y": dev(c[1]), "z": dev(c[2]), "h": dev(h0), "omega": dev(np.zeros(n))}
        H.build_neighbours(s, dev(np.minimum(h * 1.2, 0.49)), export=False)
        H.density(s)
        ok = h < 0.48
        assert np.max(np.abs(s["h"].cpu().numpy() / h - 1)[ok]) < 1e-12
        H.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_forms_of_the_solve_on_the_same_particles(hyd, precision):
    """A box of 4,000 particles alone (a warp each) and beside one of 5,000 (a
    thread each): the same lists, so the same bits in the mixed path, which sums
    in the list's order in both forms.  In FP64 a warp's lanes sum every 32nd entry
    and fold: at most 60 reordered terms, 60 2^-53 of a sum whose logarithmic slope
    in h is about three."""
    import torch
    rng = np.random.default_rng(12)
    n = (4000, 5000)
    c = rng.random((3, sum(n)))
    c[:, :2000] = 0.5 + 0.2 * (c[:, :2000] - 0.5)   # (denser in the middle of the first box)
    out = []
    for k in (1, 2):
        m = sum(n[:k])
        H = hyd.Hydro(hyd.default_config(precision=precision))
        H.set_boxes(np.concatenate([[0], np.cumsum(n[:k])]).astype(np.int64), np.ones(3 * k))
        dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")
        h0 = np.full(m, np.cbrt(24.0 / np.pi / 4000))
        s = {"x": dev(c[0, :m]), "y": dev(c[1, :m]), "z": dev(c[2, :m]), "h": dev(h0),
             "omega": dev(np.zeros(m))}
        H.build_neighbours(s, dev(np.full(m, 0.25)), export=False)
        H.density(s)
        out.append([s[q].cpu().numpy()[:n[0]] for q in ("h", "omega")])
        H.close()
    for a, b in zip(*out):
        if precision == "mixed":
            assert np.array_equal(a, b)
        else:
            assert np.max(np.abs(a / b - 1.0)) <= 3 * 60 * 2.0 ** -53


@pytest.mark.parametrize("excess", [1.0, 1e-2, 1e-4, 1e-6])
def test_step_with_n_ngb_near_the_own_term(hyd, excess):
    """FP64, N_NGB just above the 14 of a particle's own term: the neighbours add little,
    the root is flat, and its list must not be cut to a float root's margin.  The
    steps solve (few neighbours leave the matrices ill-conditioned) and agree with
    the staged solve, which cuts no list."""
    w = W.lattice_wave(16, jitter=0.1)
    H = hyd.Hydro(hyd.default_config(gamma=w["gamma"], n_ngb=14.0 + excess, max_ngb_grow=0))
    H.set_boxes(*hyd.single_box(w))
    st = hyd.to_device(w)
    for _ in range(3):
        assert H.step(st, 1e-12, check=False)["status"] in (0, -5)
    h = st["h"].clone()
    H.build_neighbours(st, h * 1.2, export=False)
    H.density(st)
    # (the slope is about 20 t^3 for one neighbour of 5 t^4 = excess / 14)
    t = min((excess / 70.0) ** 0.25, 0.3)
    tol = 1e-14 / t ** 3
    assert float((st["h"] / h - 1.0).abs().max()) < tol
    H.close()
