"""The particle order either side of its rules on size (ranking, radix tiles of
256, 1024 and 4096 keys) and with keys of more than 32 bits: a step with
sorted_output returns the stable Morton order, equal keys in the caller's
order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _key(x, y, z, L):
    q = [np.minimum((v / max(L) * 1024.0).astype(np.int64), 1023) for v in (x, y, z)]
    k = np.zeros(x.size, dtype=np.int64)
    for b in range(10):
        for a in range(3):
            k |= ((q[a] >> b) & 1) << (3 * b + 2 - a)
    return k


@pytest.mark.parametrize("sizes,L", [
    ((501,), (1, 1, 1)), ((4099,), (1, 1, 1)), ((16384,), (1, 1, 1)), ((16385,), (1, 1, 1)),
    ((77823,), (2, 1, 1)), ((311297,), (1, 1, 1)), ((2490369,), (1, 1, 1)),
    ((1000, 533, 2047), (1, 1, 1)),                 # keys of 32 bits: ranked
    ((700, 540, 900, 1201, 564), (1, 1, 1)),        # 33 bits: radix, five passes
])
def test_order_is_the_stable_morton_order(sizes, L):
    import torch
    from paper_2211_12243_gb300 import hydro
    rng = np.random.default_rng(sum(sizes))
    n = sum(sizes)
    # pairs of particles so close that their keys are equal, in a random order
    c = rng.random((3, n))
    c[:, n - n // 2:] = c[:, :n // 2] + 1e-5 / 1024
    c = c[:, rng.permutation(n)]
    x, y, z = (np.minimum(v * l, np.nextafter(l, 0)) for v, l in zip(c, L))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    box = np.repeat(np.arange(len(sizes)), sizes)
    want = np.lexsort((np.arange(n), _key(x, y, z, L), box))
    H = hydro.Hydro(hydro.default_config(precision="fp64", riemann="hllc", sorted_output=1,
                                         limiter=0, search_margin=1.5))
    H.set_boxes(off, np.tile(np.asarray(L, dtype=np.float64), len(sizes)))
    m = np.full(n, 1.0 / n)
    w = dict(x=x, y=y, z=z, m=m, px=0 * m, py=0 * m, pz=0 * m, E=1.5 * m, U=1.5 * m,
             h=np.cbrt(24.0 / np.pi * np.prod(L) / np.repeat(sizes, sizes)))
    st = hydro.to_device(w)
    rc = H.step(st, 1e-9, check=False)["status"]
    assert rc in (0, -5), rc
    assert np.array_equal(H.get_order().cpu().numpy(), want)
    H.close()
