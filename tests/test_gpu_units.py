"""The FP64 path in units far from one: the same problem with every length
scaled by a power of two, which scales every FP64 operation exactly, so that
only what passes through float can differ; and long boxes, whose float
separations are coarse against the short sides."""
import numpy as np
import pytest

from paper_2211_12243_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _scaled(w, k):
    """lengths by 2^k, masses by 8^k, velocities and pressures unchanged"""
    s = dict(w)
    for q in ("x", "y", "z", "h", "L"):
        s[q] = np.ldexp(w[q], k)
    for q in ("m", "px", "py", "pz", "E", "U"):
        s[q] = np.ldexp(w[q], 3 * k)
    return s


@pytest.mark.parametrize("name", ["wave", "lognormal"])
@pytest.mark.parametrize("k", [70, 58, -60, -74])
def test_fp64_step_in_other_length_units(name, k):
    """Two steps from rough smoothing lengths (re-searches, compacted lists):
    squares of these lengths overflow or underflow in float"""
    import torch
    from paper_2211_12243_gb300 import hydro
    w = W.lattice_wave(12, jitter=0.1) if name == "wave" else \
        W.lognormal(4099, seed=2, grid=16, contrast=100.0)
    out = []
    for kk in (0, k):
        s = _scaled(w, kk)
        H = hydro.Hydro(hydro.default_config(gamma=w["gamma"], scheme="mfm"))
        H.set_boxes(*hydro.single_box(s))
        st = hydro.to_device(s)
        stats = [H.step(st, float(np.ldexp(1e-4, kk)), check=False) for _ in range(2)]
        torch.cuda.synchronize()
        out.append((stats, {q: v.cpu().numpy() for q, v in st.items()}))
        H.close()
    (sa, a), (sb, b) = out
    for u, v in zip(sa, sb):
        for q in ("status", "grad_pairs", "flux_pairs", "ngb_rounds"):
            assert u[q] == v[q], q
    for q, e in (("h", k), ("omega", 3 * k), ("x", k), ("px", 3 * k), ("E", 3 * k)):
        c = np.ldexp(b[q], -e)
        assert np.max(np.abs(c - a[q])) <= 1e-12 * np.max(np.abs(a[q])), q


@pytest.mark.parametrize("n,k", [(4099, -66), (4099, -62), (120011, -64), (4099, 66)])
def test_lists_in_other_length_units(n, k):
    """radii whose squares are subnormal floats (or beyond them)"""
    import torch
    from paper_2211_12243_gb300 import hydro
    rng = np.random.default_rng(n)
    x, y, z = rng.random((3, n))
    hs = np.cbrt(3.0 * 40.0 / (4.0 * np.pi * n)) * rng.uniform(0.7, 1.2, n)
    out = []
    for kk in (0, k):
        H = hydro.Hydro(hydro.default_config())
        H.set_boxes(np.array([0, n], dtype=np.int64), np.full(3, np.ldexp(1.0, kk)))
        dev = lambda v: torch.as_tensor(np.ldexp(v, kk), device="cuda")
        off, idx = H.build_neighbours({"x": dev(x), "y": dev(y), "z": dev(z), "h": dev(hs)}, dev(hs))
        out.append((off.cpu().numpy(), idx.cpu().numpy()))
        H.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("length,R,h0", [(64.0, 2.3e-4, 5.7e-3), (1024.0, 1.8e-3, 6e-4)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_pairs_of_a_cluster_in_a_long_box(precision, length, R, h0):
    """A cluster whose smoothing lengths are small against the short sides of a
    long box: the fixed-point positions resolve the long side coarsely, and the
    lists that the density solve compacts must keep every member, the float
    band must not decide pairs that it cannot (the pair counts of the gradient
    and flux stages against all pairs in double)."""
    import torch
    from paper_2211_12243_gb300 import hydro
    rng = np.random.default_rng(4)
    n, L = 3000, np.array([length, 1.0, 1.0])
    d = rng.standard_normal((n, 3))
    p = 0.43 + R * d / np.linalg.norm(d, axis=1)[:, None] * np.cbrt(rng.random((n, 1)))
    p[:, 0] += 0.64 * length
    m, z = np.full(n, 1.0 / n), np.zeros(n)
    w = dict(x=p[:, 0], y=p[:, 1], z=p[:, 2], m=m, px=z, py=z, pz=z, E=1.5 * m, U=1.5 * m,
             h=np.full(n, h0))
    H = hydro.Hydro(hydro.default_config(precision=precision, max_ngb_grow=0))
    H.set_boxes(np.array([0, n], dtype=np.int64), L)
    st = hydro.to_device(w)
    s = H.step(st, 1e-12, check=False)
    torch.cuda.synchronize()
    assert s["status"] in (0, -5), s
    h = st["h"].cpu().numpy()
    assert np.median(h) < R / 3
    pairs = faces = 0
    for i in range(n):
        e = p - p[i]
        r2 = (e[:, 0] * e[:, 0] + e[:, 1] * e[:, 1]) + e[:, 2] * e[:, 2]
        r2[i] = np.inf
        mine = r2 < h[i] * h[i]
        pairs += int(np.count_nonzero(mine))
        faces += int(np.count_nonzero((mine | (r2 < h * h))[i:]))
    assert s["grad_pairs"] == pairs
    assert s["flux_pairs"] == faces
    H.close()
