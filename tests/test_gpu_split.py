"""The FP32 source iteration on the tensor cores against the equation it solves.

After a step S(n) must be the fixed point S = a P (Q + b1 S) = a P I(n) in every voxel, so
the residual a P I - S of the stored fields is formed in FP64 (P from the host tables) and
held to a bound: the stop rule leaves at most tol (1 - rho) / rho of the voxel's source, and
rounding I and S to FP32 and the FP32 sums behind them a few units of 2^-24 of it; together
below 2e-6 of max |S| of the voxel at tol = 1e-6 (1 - rho is below 0.7 where a > 0 here).
The grids leave partial 8 x 4 x 4 tiles, the optics hold vacuum, pure absorbers and thick
voxels, and the anisotropies cover a negative, an isotropic and a sharply peaked kernel.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _problem(shape, nside, g, uniform, **over):
    nx, ny, nz = shape
    p = W.homogeneous(nx, ny, nz, nside, 0.02, 8.0, g=g, steps=20, tol=1e-6)
    if not uniform:
        rng = np.random.default_rng(7)
        u = rng.random(p["mua"].shape)
        p["mua"] = (0.02 * np.exp(rng.standard_normal(u.shape))).astype(np.float32)
        p["mus"] = (8.0 * np.exp(rng.standard_normal(u.shape))).astype(np.float32)
        p["mus"][u < 0.1] = 0.0                      # pure absorbers
        p["mua"][u < 0.05] = 0.0                     # vacuum
        p["mus"][u > 0.95] = 60.0                    # thick voxels
    p["detectors"] = []
    p.update(over)
    return p


def _residual(p, steps, run=False):
    import paper_2105_01028_gb300 as T
    fw = T.Forward(p)
    rng = np.random.default_rng(1)
    I0 = np.exp(rng.standard_normal((1, fw.nv))) * (1 + 0.3 * rng.random((fw.na, fw.nv)))
    fw.set_initial_state(I0.astype(np.float32), (0.9 * I0).astype(np.float32))
    if run:
        fw.run(steps)
        fw.sync()
    else:
        fw.step(steps)
    I, S = fw.field(T.FIELD_I).astype(np.float64), fw.field(T.FIELD_S).astype(np.float64)
    status = fw.last_status
    fw.close()
    P, _ = T.phase_matrix(p["nside"], p["g"])
    mua, mus = (p[k].astype(np.float64).ravel() for k in ("mua", "mus"))
    a = np.where(mus > 0, mus / np.where(mua + mus > 0, mua + mus, 1.0), 0.0)
    r = np.max(np.abs(a * (P @ I) - S), axis=0)
    return r, np.max(np.abs(S), axis=0), status


@pytest.mark.parametrize("shape,nside,g,uniform", [
    ((8, 4, 4), 4, 0.9, True), ((9, 5, 6), 4, 0.9, False), ((12, 7, 3), 2, 0.9, False), ((20, 4, 9), 4, 0.0, False),
    ((17, 6, 5), 2, -0.6, False), ((8, 9, 4), 4, 0.99, False), ((5, 3, 2), 2, 0.3, True)])
def test_the_fields_satisfy_the_fixed_point_equation(shape, nside, g, uniform):
    r, s, status = _residual(_problem(shape, nside, g, uniform), 3)
    assert status == 0
    assert np.all(r <= 2e-6 * s + 1e-12 * s.max())


def test_the_iteration_cap_is_reported():
    import paper_2105_01028_gb300 as T
    r, s, status = _residual(_problem((9, 5, 6), 4, 0.9, False, max_iters=2), 1)
    assert status == T.W_NOT_CONVERGED


def test_a_captured_run_follows_a_change_of_anisotropy():
    import paper_2105_01028_gb300 as T
    out = []
    for first in (0.9, 0.2):
        p = _problem((12, 8, 4), 4, first, True)
        p["source"] = dict(face=4, u_mm=6.0, v_mm=4.0, half_angle_deg=30.0, pulse_steps=2, energy=1.0)
        fw = T.Forward(p)
        for g in (first, 0.2):
            fw.reset()
            assert fw.set_optics(p["mua"], p["mus"], p["nidx"], g) == 0
            fw.run(16)
            fw.sync()
        out.append(fw.field(T.FIELD_S))
        fw.close()
    assert out[0].max() > 0 and np.array_equal(out[0], out[1])
