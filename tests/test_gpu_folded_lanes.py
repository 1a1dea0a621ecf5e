"""The folded forward phase on each side of its last line, from two lanes per ray
to one, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import appga_oracle as O
from paper_2409_13344_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"
BINS = 34


@pytest.mark.parametrize("lanes", [2, 1])
@pytest.mark.parametrize("bf16", [False, True])
def test_one_and_two_lanes_against_the_oracle(lanes, bf16):
    from paper_2409_13344_gb300 import build
    build.build()
    from paper_2409_13344_gb300 import appga as A
    # one lane from 52 warps an SM of the folded half's rays on; the number of
    # angles is even, the nearest on either side (14880 at 152 SMs)
    line = 52 * 32 * torch.cuda.get_device_properties(0).multi_processor_count
    angles = 2 * (-(-line // BINS)) - (2 if lanes == 2 else 0)
    assert (angles * BINS // 2 >= line) == (lanes == 1)
    geom = W.Geometry(24, angles, BINS)
    Amat = W.siddon_matrix(geom)
    sl = W.make_slice(Amat, geom, 4.8e4, W.seed_for(3), phantom="uniform")
    ctx = A.Context(0)
    mat = A.Matrix(ctx, Amat, geom.n, angles, bf16=bf16)
    assert mat.info().quarter_turn_folded == 1
    kw = dict(max_iters=3, beta=0.1, lambda1=0.2, lambda2=0.3, eps=0.01)
    f = torch.empty(mat.d, dtype=torch.float32, device=DEV)
    p = A.default_params(a_precision=A.APPGA_PREC_BF16 if bf16 else A.APPGA_PREC_FP32, **kw)
    A.appga_reconstruct(ctx.handle, mat.handle, torch.from_numpy(sl.g).to(DEV),
                        torch.from_numpy(sl.gamma).to(DEV), None, p, f)
    if bf16:
        Amat = Amat.copy()
        Amat.data = torch.from_numpy(Amat.data).bfloat16().float().numpy()
    ref = O.appga(O.Problem(Amat, sl.g, sl.gamma, geom.n), O.Params(**kw), n_angles=angles,
                  track_phi=False).f
    # three maps; one map is within 1e-6 of the FP64 oracle at beta = 0.1
    assert np.linalg.norm(f.cpu().numpy() - ref) <= 5e-6 * np.linalg.norm(ref)
    mat.close()
    ctx.close()
