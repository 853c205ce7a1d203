"""What the FP32 iteration on the tensor cores reports: a voxel whose change is above the tolerance
when it is left counts as not converged, unless the change has sunk into the rounding of the
residual (2^-21 of the voxel's largest X, an error of amp 2^-21 in S with amp = rho / (1 - rho)).
So a call that reports success is within max(2e-6, amp 2^-20) of the fixed point.

Very thick voxels (1 - b1 down to 1e-4, eps to 1e-6: light scatters thousands of times within the
voxel) with kernels of either sign, and a start of the wrong size.
"""
import numpy as np
import pytest

import paper_2105_01028_gb300 as T
from test_gpu_split_directions import _buffers, _matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("na,g", [(48, 0.9), (192, 0.9), (192, 0.0), (192, -0.9), (48, 0.99)])
@pytest.mark.parametrize("start", [0.0, 1.0, 100.0])
def test_success_means_the_fixed_point(na, g, start):
    P32, P = _matrix(na, g)
    rng = np.random.default_rng(na)
    nvox = 260
    x = np.exp(rng.uniform(np.log(1e2), np.log(1e4), (1, nvox))) * rng.uniform(1.0, 1.6, (na, 1))
    b1 = ((x - 1 + np.exp(-x)) / x).astype(np.float32)
    eps = (10.0 ** rng.uniform(-6, -2, nvox)).astype(np.float32)
    Q = (0.5 + rng.random((na, nvox))).astype(np.float32)
    scale = 1.0 / np.mean(1.0 - (1.0 - np.float64(eps)) * b1, axis=0)
    rc, S, _ = _buffers(P32, Q, b1, eps, start * scale * Q.mean(axis=0) * np.ones((na, 1)))
    assert rc == 0
    for v in range(nvox):
        a, b = 1.0 - float(eps[v]), b1[:, v].astype(np.float64)
        ref = np.linalg.solve(np.eye(na) - a * P * b, a * (P @ Q[:, v].astype(np.float64)))
        rho = a * b.max()
        bound = max(2e-6, rho / (1.0 - rho) * 2.0 ** -20)
        assert np.max(np.abs(S[:, v] - ref)) <= bound * np.max(np.abs(ref)), v


@pytest.mark.parametrize("na", [48, 192])
def test_an_overflow_is_reported(na):
    P32, _ = _matrix(na, 0.9)
    Q = np.full((na, 140), 1.0, dtype=np.float32)
    Q[:, 7] = 3e38  # its fixed point is not an FP32 number
    b1, eps = np.full(Q.shape, 0.9), np.full(140, 0.01)
    rc, S, _ = _buffers(P32, Q, b1, eps, Q, max_iters=200)
    assert rc == T.W_NOT_CONVERGED
    # (the start's largest value sets the scale of the stop test: the others take one update)
    assert np.isfinite(np.delete(S, 7, axis=1)).all()
