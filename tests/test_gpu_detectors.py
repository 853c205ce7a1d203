"""Detectors of many voxels: the entry list (voxel x direction x detector) then spans many blocks.
A detector's curve is the sum of the curves of one-voxel detectors that cover it, entry by entry
the same products in FP64: 1e-12.  Vacuum faces and a closed box, where only the entries are left."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,boundary", [(2, "vacuum"), (4, "vacuum"), (4, "mirror")])
def test_a_wide_detector_is_the_sum_of_its_voxels(nside, boundary):
    import paper_2105_01028_gb300 as T
    p = W.homogeneous(20, 18, 6, nside, 0.01, 2.0, steps=30, tol=1e-5)
    p["boundary"] = boundary
    if boundary == "vacuum":
        p["source"] = dict(face=4, u_mm=10.0, v_mm=9.0, half_angle_deg=30.0, pulse_steps=2, energy=1.0)
    else:  # a closed box takes its light from an initial state
        p.pop("source", None)
        glow = np.random.default_rng(1).random((1, 20 * 18 * 6)) + np.zeros((12 * nside ** 2, 1))
        glow = glow.astype(np.float32)
    wide = [(9.5, 9.5, 6.0), (11.5, 8.5, 5.0), (4.5, 4.5, 3.0)]
    cells = [[(x + 0.5, y + 0.5) for y in range(18) for x in range(20)
              if (x + 0.5 - u) ** 2 + (y + 0.5 - v) ** 2 <= r * r * (1 + 1e-12)] for u, v, r in wide]
    curves = []
    for dets in ([(u, v, r) for u, v, r in wide], [(u, v, 0.5) for c in cells for u, v in c]):
        p["detectors"] = [dict(face=4, u_mm=u, v_mm=v, radius_mm=r, half_angle_deg=60.0) for u, v, r in dets]
        fw = T.Forward(W._bins(p))
        if boundary != "vacuum":
            fw.set_initial_state(glow, glow)
        fw.run(30)
        fw.sync()
        curves.append(fw.detectors())
        fw.close()
    start = 0
    for k, c in enumerate(cells):
        ref = curves[1][start:start + len(c)].sum(axis=0)
        start += len(c)
        assert ref.max() > 0
        np.testing.assert_allclose(curves[0][k], ref, rtol=1e-12, atol=0)
