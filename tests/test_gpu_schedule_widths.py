"""Launch schedules of the batched kernels by the number of slots they work on."""
import numpy as np
import pytest

from paper_2409_13344_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
GEOM = W.Geometry(61, 44, 89)
WIDTHS = (8, 16, 32)


def test_a_schedule_serves_its_own_width():
    from paper_2409_13344_gb300 import build
    build.build()
    from paper_2409_13344_gb300 import appga as A
    Amat = W.siddon_matrix(GEOM)
    ctx = A.Context(0)
    mat = A.Matrix(ctx, Amat, GEOM.n, GEOM.n_angles)
    sls = [W.make_slice(Amat, GEOM, 2e4 * (1 + i % 5), W.seed_for(3, i)) for i in range(20)]

    def served():
        # 20 requests of 3 to 15 maps in one pool of 32 slots: replays of all widths
        srv = A.Server(ctx, slots_per_pool=32, steps_per_launch=2)
        gid = srv.add_geometry(mat)
        ids = [srv.submit(gid, s.g, s.gamma, A.default_params(max_iters=3 + 12 * (i < 7), beta=0.1))
               for i, s in enumerate(sls)]
        while srv.step() != 0:
            pass
        got = [srv.collect(i) for i in ids]
        srv.close()
        return np.stack([f for f, _ in got]), np.array([st.phi_last for _, st in got])

    f0, phi0 = served()
    for k, w in enumerate(WIDTHS):
        A.appga_batch_schedule_set(mat.handle, A.appga_batch_tuning(
            K=w, a_precision=0, spmv_per_sm=3 + k, pixel_per_sm=2 + k, stencil_per_sm=1 + k,
            gather_rows_px=4 * (k % 2)))
    for K in (1, 8, 9, 16, 17, 32):
        got = A.appga_batch_schedule_get(mat.handle, K)
        k = [w >= K for w in WIDTHS].index(True)
        assert (got.spmv_per_sm, got.pixel_per_sm, got.stencil_per_sm) == (3 + k, 2 + k, 1 + k)
    assert A.appga_batch_schedule_get(mat.handle, 33).pixel_per_sm == 0
    f1, phi1 = served()
    np.testing.assert_array_equal(f1, f0)
    # the objective's double-float sums (2^-48 an addition, 4 k rows, terms of up to
    # ten times the total) are grouped by the schedule
    np.testing.assert_allclose(phi1, phi0, rtol=2e-10)
    mat.close()
    ctx.close()
