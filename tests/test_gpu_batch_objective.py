"""The objective that a batched call reports for a slice, at batch sizes on
both sides of every width of its kernels."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("bf16", [False, True])
def test_phi_does_not_depend_on_the_batch(A, bf16):
    # a row's sum is four partial sums in every width, so the double-float
    # objective of a slice is the same number in every batch
    geom = W.Geometry(61, 43, 89)
    Amat = W.siddon_matrix(geom)
    ctx = A.Context(0)
    mat = A.Matrix(ctx, Amat, geom.n, geom.n_angles, bf16=bf16)
    sls = [W.make_slice(Amat, geom, 2e4 * (1 + i % 5), W.seed_for(3, i)) for i in range(128)]
    p = A.default_params(max_iters=4, beta=0.1, track_objective=1,
                         a_precision=A.APPGA_PREC_BF16 if bf16 else A.APPGA_PREC_FP32)

    def phis(K):
        g = torch.from_numpy(np.stack([s.g for s in sls[:K]])).to(DEV)
        gam = torch.from_numpy(np.stack([s.gamma for s in sls[:K]])).to(DEV)
        f = torch.empty((K, mat.d), dtype=torch.float32, device=DEV)
        st = A.appga_reconstruct_batched(ctx.handle, mat.handle, K, g, gam, None, p, f)
        return np.array([s.phi for s in st])

    alone = phis(64)
    for K in (1, 8, 9, 17, 33, 65, 128):
        got = phis(K)
        np.testing.assert_array_equal(got[:64], alone[:min(K, 64)])
    np.testing.assert_array_equal(phis(65)[64:], phis(128)[64:65])
    mat.close()
    ctx.close()
