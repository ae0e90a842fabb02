"""Neighbour lists where the tile kernel can go wrong, against the oracle's
lists (membership r < h_search in double, bit for bit): boxes of one bucket
and of a remainder of one, radii that put whole lattice shells at the
boundary, radii too small or boxes too small for relative float coordinates,
lists longer than the fixed slots (the count-and-fill passes), and buckets
that straddle high-level Morton cells, at sizes either side of the split of
buckets among warps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hyd():
    from paper_2211_12243_gb300 import hydro
    return hydro


def _uniform(n, L, seed):
    rng = np.random.default_rng(seed)
    return [rng.random(n) * l for l in L]


def _lattice(n):
    a = (np.arange(n) + 0.5) / n
    return [v.ravel() for v in np.meshgrid(a, a, a, indexing="ij")]


def _clustered(n, seed):
    rng = np.random.default_rng(seed)
    c = rng.random((64, 3))
    p = c[rng.integers(0, 64, n)] + rng.standard_normal((n, 3)) * rng.choice([0.003, 0.03], (n, 1))
    return [np.mod(v, 1.0) * (1 - 1e-12) for v in p.T]


def _mean_h(n, L, k):
    return np.cbrt(3.0 * k * np.prod(L) / (4.0 * np.pi * n))


CASES = {
    # name: (positions, L, search radius per particle)
    "one": lambda: (_uniform(1, (1, 1, 1), 1), (1, 1, 1), np.full(1, 0.3)),
    "bucket": lambda: (_uniform(32, (1, 1, 1), 2), (1, 1, 1), np.full(32, 0.45)),
    "bucket_and_one": lambda: (_uniform(33, (1, 1, 1), 3), (1, 1, 1), np.full(33, 0.4)),
    "small_257": lambda: (_uniform(257, (1, 1, 1), 4), (1, 1, 1), np.full(257, 0.33)),
    "long_box": lambda: (_uniform(3001, (4, 1, 0.5), 5), (4, 1, 0.5),
                         np.full(3001, _mean_h(3001, (4, 1, 0.5), 40))),
    "shell_at_radius": lambda: (_lattice(20), (1, 1, 1), np.full(8000, np.sqrt(5.0) / 20)),
    "mixed_radii": lambda: (_uniform(5003, (1, 1, 1), 6), (1, 1, 1),
                            np.random.default_rng(7).uniform(1e-7, 0.12, 5003)),
    "tiny_radii": lambda: (_uniform(4099, (1, 1, 1), 8), (1, 1, 1), np.full(4099, 2e-6)),
    "long_lists": lambda: (_uniform(6007, (1, 1, 1), 9), (1, 1, 1),
                           np.full(6007, _mean_h(6007, (1, 1, 1), 180))),
    "clustered_split": lambda: (_clustered(20011, 10), (1, 1, 1),
                                np.random.default_rng(11).uniform(0.002, 0.008, 20011)),
    "clustered_whole": lambda: (_clustered(130051, 12), (1, 1, 1),
                                np.random.default_rng(13).uniform(0.001, 0.004, 130051)),
    "uniform_whole": lambda: (_uniform(120011, (1, 1, 1), 14), (1, 1, 1),
                              np.full(120011, _mean_h(120011, (1, 1, 1), 110))),
}


@pytest.mark.parametrize("name", list(CASES))
def test_lists_match_oracle(orc, hyd, name):
    import torch
    (x, y, z), L, hs = CASES[name]()
    n, L = x.size, np.asarray(L, dtype=np.float64)
    H = hyd.Hydro(hyd.default_config())
    H.set_boxes(np.array([0, n], dtype=np.int64), L)
    dev = lambda v: torch.as_tensor(np.ascontiguousarray(v, dtype=np.float64), device="cuda")
    st = {"x": dev(x), "y": dev(y), "z": dev(z), "h": dev(hs)}
    off, idx = H.build_neighbours(st, dev(hs))
    off_o, idx_o = orc.neighbours(x, y, z, L, hs)
    assert np.array_equal(off.cpu().numpy(), off_o)
    assert np.array_equal(idx.cpu().numpy(), idx_o)
    H.close()


def test_export_of_rows_longer_than_shared_memory(orc, hyd):
    import torch
    n = 1500
    x, y, z = _uniform(n, (1, 1, 1), 20)
    hs = np.full(n, 0.49)
    hs[::3] = 0.9   # (beyond half the box: nearly every particle; rows of over 1024 entries)
    H = hyd.Hydro(hyd.default_config())
    H.set_boxes(np.array([0, n], dtype=np.int64), np.ones(3))
    dev = lambda v: torch.as_tensor(np.ascontiguousarray(v, dtype=np.float64), device="cuda")
    st = {"x": dev(x), "y": dev(y), "z": dev(z), "h": dev(hs)}
    off, idx = H.build_neighbours(st, dev(hs))
    off_o, idx_o = orc.neighbours(x, y, z, np.ones(3), hs, use_grid=False)
    assert np.diff(off_o).max() > 1024
    assert np.array_equal(off.cpu().numpy(), off_o)
    assert np.array_equal(idx.cpu().numpy(), idx_o)
    H.close()


@pytest.mark.parametrize("n", [4099, 120011])
def test_radii_of_zero_and_nan_leave_the_other_lists(hyd, n):
    """A particle of radius +0, -0 or NaN has no neighbours; the lists of the
    particles that share its bucket are those of the other radii alone."""
    import torch
    x, y, z = _uniform(n, (1, 1, 1), 30)
    hs = np.full(n, _mean_h(n, (1, 1, 1), 40))
    rng = np.random.default_rng(31)
    odd = rng.choice(n, n // 50, replace=False)
    out = []
    for special in (False, True):
        r = hs.copy()
        r[odd] = np.resize([-0.0, np.nan, 0.0], odd.size) if special else 1e-9
        H = hyd.Hydro(hyd.default_config())
        H.set_boxes(np.array([0, n], dtype=np.int64), np.ones(3))
        dev = lambda v: torch.as_tensor(np.ascontiguousarray(v, dtype=np.float64), device="cuda")
        st = {"x": dev(x), "y": dev(y), "z": dev(z), "h": dev(hs)}
        off, idx = H.build_neighbours(st, dev(r))
        out.append((off.cpu().numpy(), idx.cpu().numpy()))
        H.close()
    (oa, ia), (ob, ib) = out
    ca, cb = np.diff(oa), np.diff(ob)
    assert np.all(cb[odd] == 0) and np.all(ca[odd] == 1)      # (the particle itself)
    ca[odd] = 0
    assert np.array_equal(ca, cb)
    keep = np.ones(ia.size, dtype=bool)
    keep[oa[odd]] = False
    assert np.array_equal(ia[keep], ib)
