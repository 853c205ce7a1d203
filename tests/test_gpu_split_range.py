"""The FP32 iteration on the tensor cores over FP32's range: the equation is linear, and a power of
two that multiplies every input multiplies every output, exactly, as long as nothing leaves the
range of FP32 numbers.  Buffers: the same bits times that power.  Whole solves and gradients at
2^-110 and 2^-100: gradual underflow begins 2^-26 below values of one, so voxels (directions)
within 1e-3 of the largest are held to 1e-6 of theirs; the gradient, whose tails underflow
inside the sums, to 1e-5 of its largest entry.
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_adjoint import _gpu_gradient, _problem as _adjoint_problem
from test_gpu_split_directions import _buffers, _matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("na", [48, 192])
@pytest.mark.parametrize("power", [-100, -84, -60, 60, 113])
def test_buffers_scale_with_their_inputs(na, power):
    P32, _ = _matrix(na, 0.9)
    rng = np.random.default_rng(na)
    nvox = 300
    x = np.exp(rng.uniform(np.log(0.1), np.log(20.0), (1, nvox))) * rng.uniform(1.0, 1.6, (na, 1))
    b1 = ((x - 1 + np.exp(-x)) / x).astype(np.float32)
    eps = (10.0 ** rng.uniform(-3, 0, nvox)).astype(np.float32)
    Q = (0.5 + rng.random((na, nvox))).astype(np.float32)
    S0 = (Q * (0.5 + rng.random((1, nvox)))).astype(np.float32)
    Q[:, ::3] *= np.float32(2.0 ** -10)  # dim and bright voxels in one tile
    f = np.float32(2.0 ** power)
    rc, S, I = _buffers(P32, Q, b1, eps, S0)
    rc2, S2, I2 = _buffers(P32, Q * f, b1, eps, S0 * f)
    assert rc == rc2 == 0 and np.isfinite(S2).all()
    assert np.array_equal(S2, S * f) and np.array_equal(I2, I * f)


@pytest.mark.parametrize("nside,uniform", [(2, False), (4, True), (4, False)])
def test_a_dim_source_gives_the_same_fields(nside, uniform):
    import paper_2105_01028_gb300 as T
    p = W.homogeneous(12, 9, 8, nside, 0.02, 2.0, g=0.9, steps=12, tol=1e-6)
    if not uniform:
        p["mus"] = (2.0 * (1.0 - 0.5 * np.random.default_rng(3).random(p["mus"].shape))).astype(np.float32)
    p["detectors"] = []
    out = []
    for power in (0, -110):
        p["source"] = dict(face=4, u_mm=6.0, v_mm=4.0, half_angle_deg=30.0, pulse_steps=2, energy=2.0 ** power)
        fw = T.Forward(p)
        fw.step(12)
        out.append(fw.field(T.FIELD_S).astype(np.float64) * 2.0 ** -power)
        fw.close()
    big = np.max(out[0], axis=0) > 1e-3 * out[0].max()
    assert big.sum() > 100
    assert np.all(np.abs(out[1] - out[0])[:, big] <= 1e-6 * np.max(out[0], axis=0)[big])


@pytest.mark.parametrize("shape,nside", [((6, 6, 6), 2), ((8, 8, 6), 4)])
def test_gradients_of_a_misfit_in_absolute_units(shape, nside):
    p = _adjoint_problem(*shape, nside, 16, False)
    G = 0.5 + np.random.default_rng(3).random((len(p["detectors"]), p["nbins"]))
    _, ga, gs = _gpu_gradient(p, 16, 5, G)
    _, ga2, gs2 = _gpu_gradient(p, 16, 5, G * 2.0 ** -100)
    for a, b in ((ga, ga2), (gs, gs2)):
        assert np.max(np.abs(b * 2.0 ** 100 - a)) <= 1e-5 * np.max(np.abs(a))
