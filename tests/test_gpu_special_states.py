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
