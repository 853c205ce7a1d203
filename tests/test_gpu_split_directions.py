"""The FP32 iteration on the tensor cores direction by direction: what goes into a weak direction
is held to its own size, not to the voxel's brightest direction.

The call on caller-owned buffers with b1 = 0 and eps = 0 returns S = P Q, one product, so that
each direction can be compared with FP64 (P with its diagonal made so that the rows sum to one,
as the call does).

One bright direction (a power of two, so that it splits exactly) asks for a column of P: an entry
is held to 1.5e-8 of itself by its three FP16 terms (1.2e-7 where it is below 1e-4 of the largest:
g = -0.95), the two accumulators are added with three FP32 roundings of 2^-24: 4e-7.

A row in which one direction outshines the others by up to 1e6: products of third terms that are
left out and the accumulator's truncation are 6.5e-7 of the weakest output at most (emulated in
FP64), four FP32 roundings 2.4e-7: 1.5e-6 is asked for (a sum of 192 FP32 products in turn:
2.9e-6; two terms per factor: 2.8e-4).  The same through a context, in a thin medium (b1 below
0.006, tolerance at the floor): the residual a P I - S of the stored fields in each direction,
with the stored I and S rounded and two outer residuals' error in it: 3e-6 of S.

A start far above the result, in voxels so thin that one update reaches the fixed point: the bar of
one product, 1.5e-6, as the start's rounding (2^-24 of it) must not stay in the result.
"""
import ctypes

import numpy as np
import pytest

import workloads as W

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


@pytest.mark.parametrize("na,g", [(48, 0.9), (192, 0.9), (192, 0.99)])
@pytest.mark.parametrize("weak", [1.0, 1e-2, 1e-4, 1e-6])
def test_weak_directions_beside_a_bright_one(na, g, weak):
    P32, P = _matrix(na, g)
    rng = np.random.default_rng(na)
    nvox = 300
    Q = (weak * rng.random((na, nvox))).astype(np.float32)
    Q[rng.integers(0, na, nvox), np.arange(nvox)] = 1.0 - 0.4 * rng.random(nvox)
    z = np.zeros_like(Q)
    rc, S, _ = _buffers(P32, Q, z, np.zeros(nvox), z)
    assert rc == 0
    ref = P @ Q.astype(np.float64)
    assert np.all(np.abs(S - ref) <= 1.5e-6 * np.abs(ref))


@pytest.mark.parametrize("nside,uniform", [(2, True), (4, True), (4, False)])
def test_weak_directions_of_a_step(nside, uniform):
    import paper_2105_01028_gb300 as T
    p = W.homogeneous(12, 9, 8, nside, 0.001, 0.01, g=0.9, steps=4, tol=1e-12)
    rng = np.random.default_rng(nside)
    if not uniform:
        p["mus"] = (0.01 * (1.0 - 0.5 * rng.random(p["mus"].shape))).astype(np.float32)
    p["detectors"] = []
    fw = T.Forward(p)
    I0 = np.repeat(1e-4 * rng.random((fw.na, 1)), fw.nv, axis=1)
    I0[5] = 1.0
    fw.set_initial_state(I0.astype(np.float32), np.zeros_like(I0, dtype=np.float32))
    fw.step(1)
    I, S = fw.field(T.FIELD_I).astype(np.float64), fw.field(T.FIELD_S).astype(np.float64)
    fw.close()
    P, _ = T.phase_matrix(nside, 0.9)
    mua, mus = (p[k].astype(np.float64).ravel() for k in ("mua", "mus"))
    ref = mus / (mua + mus) * (P @ I)
    assert ref.min() > 0 and ref.max() > 300 * ref.min()
    assert np.all(np.abs(ref - S) <= 3e-6 * ref)


@pytest.mark.parametrize("na", [48, 192])
@pytest.mark.parametrize("b1", [0.0, 1e-9])
@pytest.mark.parametrize("start", [1e4, 1e9])
def test_nothing_of_a_bright_start_is_left(na, b1, start):
    P32, P = _matrix(na, 0.9)
    rng = np.random.default_rng(na)
    nvox = 200
    Q = (0.5 + rng.random((na, nvox))).astype(np.float32)
    S0 = (start * rng.random((na, nvox))).astype(np.float32)
    rc, S, _ = _buffers(P32, Q, np.full(Q.shape, b1), np.zeros(nvox), S0)
    assert rc == 0
    ref = np.linalg.solve(np.eye(na) - np.float64(np.float32(b1)) * P, P @ Q.astype(np.float64))
    assert np.all(np.abs(S - ref) <= 1.5e-6 * np.abs(ref))
