"""Team widths, row deals and stencil runs of the batched kernels at the sizes
where they can go wrong: numbers of slices around every width, image sides
around the stencil's column strips and row runs, rays that do not divide by
the angles' tiles."""
import numpy as np
import pytest

from oracle import appga_oracle as O
from paper_2409_13344_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


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


def run(A, ctx, mat, sls, **kw):
    K = len(sls)
    g = torch.from_numpy(np.stack([s.g for s in sls])).to(DEV)
    gam = torch.from_numpy(np.stack([s.gamma for s in sls])).to(DEV)
    f = torch.empty((K, mat.d), dtype=torch.float32, device=DEV)
    A.appga_reconstruct_batched(ctx.handle, mat.handle, K, g, gam, None, A.default_params(**kw), f)
    return f.cpu().numpy()


@pytest.mark.parametrize("bf16", [False, True])
def test_width_never_changes_a_slice(A, ctx, bf16):
    # a row's sum is four partial sums whatever the team's width: the same
    # slices in batches of any size give the same images bit for bit
    geom = W.Geometry(33, 21, 47)  # odd everything: ragged packs, tiles and rounds
    Amat = W.siddon_matrix(geom)
    mat = A.Matrix(ctx, Amat, geom.n, geom.n_angles, bf16=bf16)
    sls = [W.make_slice(Amat, geom, 2e4 * (1 + i % 5), W.seed_for(3, i)) for i in range(128)]
    kw = dict(max_iters=6, beta=0.1,
              a_precision=A.APPGA_PREC_BF16 if bf16 else A.APPGA_PREC_FP32)
    whole = run(A, ctx, mat, sls, **kw)
    for K in (1, 7, 8, 9, 16, 17, 32, 33, 64, 65):
        np.testing.assert_array_equal(run(A, ctx, mat, sls[:K], **kw), whole[:K])


@pytest.mark.parametrize("n,angles,bins", [(1, 4, 3), (3, 5, 7), (27, 16, 41), (28, 15, 43),
                                           (29, 18, 45), (57, 12, 83)])
def test_against_the_oracle_at_tile_edges(A, ctx, n, angles, bins):
    # three maps; one map is within 1e-6 of the FP64 oracle at beta = 0.1
    geom = W.Geometry(n, angles, bins)
    Amat = W.siddon_matrix(geom)
    mat = A.Matrix(ctx, Amat, geom.n, geom.n_angles)
    sls = [W.make_slice(Amat, geom, 300.0 * n * (i + 1), W.seed_for(3, i), phantom="uniform")
           for i in range(3)]
    f = run(A, ctx, mat, sls, max_iters=3, beta=0.1, lambda1=0.2, lambda2=0.3, eps=0.01)
    for i, sl in enumerate(sls):
        prob = O.Problem(Amat, sl.g, sl.gamma, geom.n)
        ref = O.appga(prob, O.Params(max_iters=3, beta=0.1, lambda1=0.2, lambda2=0.3, eps=0.01),
                      n_angles=angles, track_phi=False)
        err = np.linalg.norm(f[i] - ref.f)
        assert err <= 5e-6 * np.linalg.norm(ref.f), (i, err)


def test_row_orders_of_a_matrix_without_angle_tiles(A, ctx):
    # m not a multiple of the angles: rays in ascending order, the same problem
    geom = W.Geometry(20, 10, 31)
    Amat = W.siddon_matrix(geom)[:-3]
    rng = np.random.default_rng(5)
    g = rng.poisson(20.0, (2, Amat.shape[0])).astype(np.float32)
    gam = np.full_like(g, 2.0)
    mat = A.Matrix(ctx, Amat, geom.n, geom.n_angles)
    f = torch.empty((2, mat.d), dtype=torch.float32, device=DEV)
    A.appga_reconstruct_batched(ctx.handle, mat.handle, 2, torch.from_numpy(g).to(DEV),
                                torch.from_numpy(gam).to(DEV), None,
                                A.default_params(max_iters=3, beta=0.1), f)
    for i in range(2):
        ref = O.appga(O.Problem(Amat, g[i], gam[i], geom.n), O.Params(max_iters=3, beta=0.1),
                      n_angles=geom.n_angles, track_phi=False)
        err = np.linalg.norm(f[i].cpu().numpy() - ref.f)
        assert err <= 5e-6 * np.linalg.norm(ref.f), (i, err)
