"""The FP32 iteration on the tensor cores direction by direction: what goes into a weak direction
is held to its own size, not to the voxel's brightest direction.

The call on caller-owned buffers with b1 = 0 and eps = 0 returns S = P Q, one product, so that
each direction can be compared with FP64 (P with its diagonal made so that the rows sum to one,
as the call does).

One bright direction (a power of two, so that it splits exactly) asks for a column of P: an entry
is held to 1.5e-8 of itself by its three FP16 terms (1.2e-7 where it is below 1e-4 of the largest:
g = -0.95), the two accumulators are added with three FP32 roundings of 2^-24: 4e-7.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _buffers(P32, Q, b1, eps, S0, tol=1e-6, max_iters=5000):
    """(rc, S, I) of the call that allocates nothing."""
    torch = pytest.importorskip("torch")
    import paper_2105_01028_gb300 as T
    na, nvox = Q.shape
    d = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).cuda() for v in (P32, Q, b1, eps, S0)]
    S, I = torch.empty_like(d[1]), torch.empty_like(d[1])
    fn = T.lib().trinity_source_iteration_noalloc
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 7 + [ctypes.c_double, ctypes.c_int,
                                                                          ctypes.POINTER(ctypes.c_int), ctypes.c_void_p]
    rc = fn(na, nvox, *(t.data_ptr() for t in d), S.data_ptr(), I.data_ptr(), tol, max_iters, None, None)
    return rc, S.cpu().numpy(), I.cpu().numpy()


def _matrix(na, g):
    import paper_2105_01028_gb300 as T
    P32 = T.phase_matrix(int(round((na / 12) ** 0.5)), g)[0].astype(np.float32)
    P = P32.astype(np.float64)
    np.fill_diagonal(P, 0.0)
    np.fill_diagonal(P, 1.0 - P.sum(axis=1))
    return P32, P


@pytest.mark.parametrize("na,g", [(48, 0.9), (192, 0.9), (192, 0.99), (192, 0.0), (48, -0.95), (192, -0.95)])
def test_every_entry_of_the_phase_matrix_counts(na, g):
    P32, P = _matrix(na, g)
    Q = np.zeros((na, na + 3))
    Q[np.arange(na + 3) % na, np.arange(na + 3)] = 2.0 ** (np.arange(na + 3) % 7 - 3)
    z = np.zeros_like(Q)
    rc, S, _ = _buffers(P32, Q, z, np.zeros(na + 3), z)
    assert rc == 0
    ref = P @ Q
    assert np.all(np.abs(S - ref) <= 4e-7 * np.abs(ref))
