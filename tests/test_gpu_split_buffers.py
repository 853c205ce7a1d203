"""The source iteration on caller-owned buffers against its fixed point in FP64.

S = (1 - eps) P (Q + b1 S) is solved in FP64 per voxel (dense, P with its diagonal made so
that the rows sum to one, as the call does).  Bound: the stop rule leaves at most tol =
1e-6 of max |S| of the voxel, FP32 rounding of the sums amplified by the scattering a few
1e-7: 2e-6 of the voxel's max |S|.  Sizes: one voxel, a partial and a full 128-voxel tile
with a remainder, more tiles than SMs; kernels with positive, zero and negative mean cosine.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("na,nvox,g", [(48, 1, 0.9), (192, 100, 0.9), (192, 129, -0.7), (48, 257, 0.0),
                                       (192, 20001, 0.9), (48, 20011, 0.6)])
def test_buffers_hold_the_fixed_point(na, nvox, g):
    torch = pytest.importorskip("torch")
    import paper_2105_01028_gb300 as T
    rng = np.random.default_rng(nvox)
    nside = int(round((na / 12) ** 0.5))
    P32 = T.phase_matrix(nside, g)[0].astype(np.float32)
    mut = np.exp(rng.uniform(np.log(0.05), np.log(40.0), nvox))
    eps = (10.0 ** rng.uniform(-4, 0, nvox)).astype(np.float32)
    eps[rng.random(nvox) < 0.1] = 1.0
    ds = 1.0 / np.max(np.abs(T.healpix_dirs(nside)), axis=1)
    x = ds[:, None] * mut[None, :]
    b1 = ((x - 1 + np.exp(-x)) / x).astype(np.float32)
    Q = (np.exp(rng.standard_normal((1, nvox))) * rng.random((na, nvox))).astype(np.float32)
    S0 = (Q.mean(axis=0, keepdims=True) * (1 + rng.random((na, nvox)))).astype(np.float32)
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in
         dict(P=P32, Q=Q, b1=b1, eps=eps, S0=S0).items()}
    S, I = torch.empty_like(d["Q"]), torch.empty_like(d["Q"])
    fn = T.lib().trinity_source_iteration_noalloc
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 7 + [ctypes.c_double, ctypes.c_int,
                                                                          ctypes.POINTER(ctypes.c_int), ctypes.c_void_p]
    it = ctypes.c_int(0)
    rc = fn(na, nvox, d["P"].data_ptr(), d["Q"].data_ptr(), d["b1"].data_ptr(), d["eps"].data_ptr(), d["S0"].data_ptr(),
            S.data_ptr(), I.data_ptr(), 1e-6, 5000, ctypes.byref(it), None)
    assert rc == 0 and it.value >= 1
    S, I = S.cpu().numpy().astype(np.float64), I.cpu().numpy()
    Pd = P32.astype(np.float64)
    Pd += np.diag(1.0 - Pd.sum(axis=1))
    pick = np.unique(np.r_[0, nvox - 1, rng.integers(0, nvox, 150)])
    for v in pick:
        a = 1.0 - float(eps[v])
        ref = np.linalg.solve(np.eye(na) - a * Pd * b1[:, v].astype(np.float64), a * (Pd @ Q[:, v].astype(np.float64)))
        assert np.max(np.abs(S[:, v] - ref)) <= 2e-6 * np.max(np.abs(ref)) + 1e-30, v
    assert np.array_equal(I, np.asarray(np.float64(b1) * S + Q, dtype=np.float32)) or \
        np.max(np.abs(I - (b1 * S + Q))) <= 2.0 ** -23 * np.max(np.abs(I))
