"""A captured step and the layout of the boxes: hydro_set_boxes may keep the
numbers of particles, buckets and tree levels and still change the number of
boxes and the size of every level, which the captured kernels hold by value.
Each step is compared with the same step of a context that has seen no other
layout."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# equal numbers of particles (512), buckets (16) and levels (2)
THREE = (np.array([0, 256, 384, 512], dtype=np.int64),
         np.array([1.0, 1, 1, 2.0, 2, 2, 2.0, 2, 2]))
TWO = (np.array([0, 256, 512], dtype=np.int64), np.array([1.0, 1, 1, 2.0, 2, 2]))


def _state(boxes):
    off, L = boxes
    rng = np.random.default_rng(int(off.size))
    n = int(off[-1])
    box = np.repeat(np.arange(off.size - 1), np.diff(off))
    l = L.reshape(-1, 3)[box]
    x, y, z = (rng.random((n, 3)) * l).T
    m = np.full(n, 1.0 / n)
    u = 1.5 + 0.2 * rng.random(n)
    v = 0.1 * rng.standard_normal((3, n))
    h = np.cbrt(3 * 24.0 / (4 * np.pi) * l.prod(1) / np.diff(off)[box])
    return dict(x=x, y=y, z=z, m=m, px=m * v[0], py=m * v[1], pz=m * v[2], U=m * u,
                E=m * (u + 0.5 * (v * v).sum(0)), h=h)


def _context(hydro, precision):
    return hydro.Hydro(hydro.default_config(precision=precision, n_ngb=24.0))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
def test_steps_follow_a_change_of_the_boxes(precision, tol):
    import torch
    from paper_2211_12243_gb300 import hydro
    dt = 1e-4
    H = _context(hydro, precision)
    H.set_boxes(*THREE)      # (the buffers hold the larger layout from here on)
    H.reserve(512, 256)      # (no list outgrows its slots: the same buffers throughout)
    st = hydro.to_device(_state(THREE))
    for step, boxes in enumerate((THREE, TWO, THREE, TWO, THREE)):
        H.set_boxes(*boxes)
        w = _state(boxes)
        for k, v in w.items():
            st[k].copy_(torch.as_tensor(v))
        s = H.step(st, dt, check=False)
        assert s["graph"] == (1 if step else 0)
        F = _context(hydro, precision)
        F.set_boxes(*boxes)
        sf = hydro.to_device(w)
        f = F.step(sf, dt, check=False)
        torch.cuda.synchronize()
        for k in ("status", "grad_pairs", "flux_pairs"):
            assert s[k] == f[k], (k, s[k], f[k])
        for k in ("h", "omega", "px", "E"):
            a, b = st[k].cpu().numpy(), sf[k].cpu().numpy()
            assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)), k
        F.close()
    H.close()
