"""The FP32 iteration at 192 directions where a CTA takes several tiles of 128 voxels, so that
what one tile leaves behind (ring slots and their parities, weight tables, staged operands,
reduction buffers) is there when the next one starts.  Forward fields: the residual bound of
test_gpu_split.py, on 400 tiles with TMA stores (nx a multiple of 4) and 480 with plain ones
(nx odd), with optics that vary.  Gradient: the bars of test_gpu_adjoint.py against the FP64
oracle on 165 tiles (152 SMs), the pulse in the tiles that are second in their CTA, one
detector over the whole face so that the adjoint field reaches every tile.
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_adjoint import _compare, _gpu_gradient, _oracle_gradient
from test_gpu_split import _problem, _residual

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [40, 41])
def test_the_fixed_point_holds_over_many_tiles(nx):
    r, s, status = _residual(_problem((nx, 40, 32), 4, 0.9, False), 2)
    assert status == 0
    assert np.all(r <= 2e-6 * s + 1e-12 * s.max())


def test_gradients_over_many_tiles_match_the_oracle():
    p = W.homogeneous(5, 42, 60, 4, 0.05, 2.0, steps=8, tol=1e-6)
    rng = np.random.default_rng(5)
    p["mua"] = (0.05 * (1 + 0.5 * rng.random(p["mua"].shape))).astype(np.float32)
    p["mus"] = (2.0 * (1 + 0.5 * rng.random(p["mus"].shape))).astype(np.float32)
    p["max_iters"] = 5000
    p["source"] = dict(face=0, u_mm=20.0, v_mm=57.0, half_angle_deg=30.0, pulse_steps=2, energy=1.0)
    p["detectors"] = [dict(face=0, u_mm=21.0, v_mm=30.0, radius_mm=60.0, half_angle_deg=60.0)]
    p = W._bins(p)
    _, ga_ref, gs_ref, E = _oracle_gradient(p, 8, np.zeros((1, p["nbins"])))
    _, ga, gs = _gpu_gradient(p, 8, 3, E)
    lit = np.abs(ga_ref).reshape(60, -1).max(axis=1) > 1e-6 * np.abs(ga_ref).max()  # along z
    assert lit[56:].any()  # 11 tiles to every four voxels along z: tiles 154 to 164
    _compare(ga, ga_ref)
    _compare(gs, gs_ref)
