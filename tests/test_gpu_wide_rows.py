"""A matrix whose rows are strips of 40 pixels, through the layout of the solver
loop and against the FP64 oracle."""
import numpy as np
import pytest

from oracle import appga_oracle as O
from test_matrix_layout_cpu import strips

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("bf16", [False, True])
def test_wide_rows_keep_the_sliced_layout(bf16):
    from paper_2409_13344_gb300 import build
    build.build()
    from paper_2409_13344_gb300 import appga as A
    n, angles = 256, 4
    Amat = strips(n, angles, 13, 20.0, 40)
    Amat.sort_indices()
    rng = np.random.default_rng(1)
    truth = rng.random(n * n) * 0.1
    gam = np.full(Amat.shape[0], 2.0, np.float32)
    g = rng.poisson(Amat @ truth + gam).astype(np.float32)
    ctx = A.Context(0)
    mat = A.Matrix(ctx, Amat, n, angles, bf16=bf16)
    assert mat.info().sliced_layout == 1
    kw = dict(max_iters=3, beta=0.1, lambda1=0.2, lambda2=0.3, eps=0.01)
    f = torch.empty(mat.d, dtype=torch.float32, device=DEV)
    p = A.default_params(a_precision=A.APPGA_PREC_BF16 if bf16 else A.APPGA_PREC_FP32, **kw)
    A.appga_reconstruct(ctx.handle, mat.handle, torch.from_numpy(g).to(DEV),
                        torch.from_numpy(gam).to(DEV), None, p, f)
    ref_mat = Amat.copy()
    if bf16:
        ref_mat.data = torch.from_numpy(Amat.data).bfloat16().float().numpy()
    ref = O.appga(O.Problem(ref_mat, g, gam, n), O.Params(**kw), n_angles=angles,
                  track_phi=False).f
    # three maps; one map is within 1e-6 of the FP64 oracle at beta = 0.1
    assert np.linalg.norm(f.cpu().numpy() - ref) <= 5e-6 * np.linalg.norm(ref)
    mat.close()
    ctx.close()
