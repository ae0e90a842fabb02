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
