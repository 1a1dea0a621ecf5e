"""Device memory of the server's pools: what a pool holds, and admission where
it is short."""
import numpy as np
import pytest

from paper_2409_13344_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
GEOM = W.Geometry(128, 90, 185)


@pytest.fixture(scope="module")
def A():
    from paper_2409_13344_gb300 import build
    build.build()
    from paper_2409_13344_gb300 import appga
    if not torch.cuda.is_available():
        pytest.fail("the -m gpu tests need a CUDA device")
    return appga


@pytest.fixture(scope="module")
def ctx(A):
    c = A.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def problem():
    Amat = W.siddon_matrix(GEOM)
    return Amat, [W.make_slice(Amat, GEOM, 2e5 * (1 + i % 3), W.seed_for(3, i)) for i in range(6)]


def budget(Amat, slots):
    # seven image and seven sinogram vectors a slot (iterates, projections,
    # inputs) and the objective's partial sums (16 bytes per slot and block)
    m, d = Amat.shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 4 * slots * 7 * (m + d) + 16 * slots * (32 * sms + 64)


def test_a_pool_fits_seven_images_and_sinograms_a_slot(A, ctx, problem):
    Amat, sls = problem
    mat = A.Matrix(ctx, Amat, GEOM.n, GEOM.n_angles)
    rng = np.random.default_rng(0)
    f0 = [None if i % 2 else rng.random(mat.d, dtype=np.float32) for i in range(6)]

    def serve(jobs):
        srv = A.Server(ctx, slots_per_pool=32, steps_per_launch=4,
                       hbm_budget_bytes=budget(Amat, 32))
        gid = srv.add_geometry(mat)
        ids = [srv.submit(gid, sls[i].g, sls[i].gamma, A.default_params(max_iters=k, beta=0.1),
                          f0[i]) for i, k in jobs]
        for _ in range(1000):
            if srv.step() == 0:
                break
        assert srv.summary().completed == len(jobs)
        out = [srv.collect(i)[0] for i in ids]
        srv.close()
        return out

    # more requests than slots: images retired and admitted between replays, with
    # and without an initial image, equal those of the same requests alone
    jobs = [(i % 6, 3 + (5 * i) % 11) for i in range(48)]
    mixed = serve(jobs)
    for job in sorted(set(jobs))[::5]:
        alone = serve([job])[0]
        for j, f in zip(jobs, mixed):
            if j == job:
                np.testing.assert_array_equal(f, alone)
    mat.close()


def test_the_first_pool_counts_the_matrix_layout(A, ctx, problem):
    # with free memory that holds a pool's slots but not the layout its kernels
    # stream (at least 10 bytes an entry: 20 a column of a block of four rows, A
    # and A^T), the request waits, and runs once there is room
    Amat, sls = problem
    mat = A.Matrix(ctx, Amat, GEOM.n, GEOM.n_angles)
    before = mat.info().device_bytes
    hold = torch.empty(1 << 30, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    srv = A.Server(ctx, slots_per_pool=32,
                   hbm_reserve_bytes=free - budget(Amat, 32) - 5 * Amat.nnz)
    gid = srv.add_geometry(mat)
    rid = srv.submit(gid, sls[0].g, sls[0].gamma, A.default_params(max_iters=3, beta=0.1))
    for _ in range(3):
        assert srv.step() == 1
    assert srv.summary().pools == 0
    assert mat.info().device_bytes - before < 1 << 20
    del hold
    torch.cuda.empty_cache()
    for _ in range(100):
        if srv.step() == 0:
            break
    assert srv.summary().completed == 1 and srv.summary().pools == 1
    assert mat.info().device_bytes - before >= 10 * Amat.nnz
    srv.collect(rid)
    srv.close()
    mat.close()
