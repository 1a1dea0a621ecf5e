"""The batched stencil where FP32 squares overflow: eps beyond 1.8e19 (the
quadratic limit, with weights as large) and difference fields beyond it."""
import numpy as np
import pytest

from oracle import appga_oracle as O
from paper_2409_13344_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"
GEOM = W.Geometry(29, 18, 45)


@pytest.fixture(scope="module")
def A():
    from paper_2409_13344_gb300 import build
    build.build()
    from paper_2409_13344_gb300 import appga
    if not torch.cuda.is_available():
        pytest.fail("the -m gpu tests need a CUDA device")
    return appga


@pytest.fixture(scope="module")
def mat(A):
    c = A.Context(0)
    m = A.Matrix(c, W.siddon_matrix(GEOM), GEOM.n, GEOM.n_angles)
    yield m
    m.close()
    c.close()


def batched(A, mat, g, gam, f0, **kw):
    f = torch.empty((len(g), mat.d), dtype=torch.float32, device=DEV)
    A.appga_reconstruct_batched(mat.ctx.handle, mat.handle, len(g), torch.from_numpy(g).to(DEV),
                                torch.from_numpy(gam).to(DEV),
                                None if f0 is None else torch.from_numpy(f0).to(DEV),
                                A.default_params(**kw), f)
    return f.cpu().numpy()


@pytest.mark.parametrize("eps", [1e18, 1.8e19, 1.9e19, 1e20, 1e25, 1e37])
def test_quadratic_limit_against_the_oracle(A, mat, eps):
    # three maps; one map is within 1e-6 of the FP64 oracle at beta = 0.1
    Amat = W.siddon_matrix(GEOM)
    sls = [W.make_slice(Amat, GEOM, 1e4 * (i + 1), W.seed_for(3, i), phantom="uniform")
           for i in range(2)]
    kw = dict(max_iters=3, beta=0.1, lambda1=0.1 * eps, lambda2=0.05 * eps, eps=eps)
    f = batched(A, mat, np.stack([s.g for s in sls]), np.stack([s.gamma for s in sls]), None, **kw)
    for i, sl in enumerate(sls):
        ref = O.appga(O.Problem(Amat, sl.g, sl.gamma, GEOM.n), O.Params(**kw),
                      n_angles=GEOM.n_angles, track_phi=False).f
        assert np.linalg.norm(f[i] - ref) <= 5e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("eps", [1e-3, 1e20])
def test_overflowing_fields_as_in_the_single_slice_call(A, mat, eps):
    # |u|^2 is infinite in FP32: the gradient of such a group is zero in both
    rng = np.random.default_rng(4)
    m, d = W.siddon_matrix(GEOM).shape
    f0 = (3e20 * rng.random(d)).astype(np.float32)
    g, gam = rng.poisson(20.0, m).astype(np.float32), np.full(m, 2.0, np.float32)
    kw = dict(max_iters=3, beta=0.1, lambda1=1.0, lambda2=0.5, eps=eps)
    one = torch.empty(d, dtype=torch.float32, device=DEV)
    A.appga_reconstruct(mat.ctx.handle, mat.handle, torch.from_numpy(g).to(DEV),
                        torch.from_numpy(gam).to(DEV), torch.from_numpy(f0).to(DEV),
                        A.default_params(**kw), one)
    one = one.cpu().numpy().astype(np.float64)
    f = batched(A, mat, g[None], gam[None], f0[None], **kw)[0]
    assert np.linalg.norm(f - one) <= 5e-6 * np.linalg.norm(one)
