"""Lanes per row of the single-slice sliced layout and groups per row block of
the batched one, at matrix sizes on each side of every line of their rules,
against the FP64 oracle."""
import numpy as np
import pytest

from oracle import appga_oracle as O
from paper_2409_13344_gb300 import workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"
PAR = dict(max_iters=3, beta=0.1, lambda1=0.2, lambda2=0.3, eps=0.01)


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


# The pixel phase has 1 / 2 / 4 lanes per row from 121600 / 60800 / 30400
# pixels, the forward phase from 252928 / 126464 / 63232 rays (152 SMs), half
# of them where the matrix is folded (even image side and angles).
@pytest.mark.parametrize("n,angles,bins", [(178, 6, 253), (247, 5, 350), (350, 4, 497),
                                           (24, 1872, 34), (24, 3734, 34), (24, 7484, 34),
                                           (23, 7485, 34)])
@pytest.mark.parametrize("bf16", [False, True])
def test_lanes_against_the_oracle(A, ctx, n, angles, bins, bf16):
    # three maps; one map is within 1e-6 of the FP64 oracle at beta = 0.1
    geom = W.Geometry(n, angles, bins)
    Amat = W.siddon_matrix(geom)
    sl = W.make_slice(Amat, geom, 2000.0 * n, W.seed_for(3), phantom="uniform")
    mats = [A.Matrix(ctx, Amat, n, angles, bf16=bf16)]
    if mats[0].info().quarter_turn_folded:
        mats.append(A.Matrix(ctx, Amat, n, angles, bf16=bf16, fold=False))
    if bf16:
        Amat = Amat.copy()
        Amat.data = torch.from_numpy(Amat.data).bfloat16().float().numpy()
    ref = O.appga(O.Problem(Amat, sl.g, sl.gamma, n), O.Params(**PAR), n_angles=angles,
                  track_phi=False).f
    for mat in mats:
        f = torch.empty(mat.d, dtype=torch.float32, device=DEV)
        p = A.default_params(a_precision=A.APPGA_PREC_BF16 if bf16 else A.APPGA_PREC_FP32, **PAR)
        A.appga_reconstruct(ctx.handle, mat.handle, torch.from_numpy(sl.g).to(DEV),
                            torch.from_numpy(sl.gamma).to(DEV), None, p, f)
        err = np.linalg.norm(f.cpu().numpy() - ref)
        assert err <= 5e-6 * np.linalg.norm(ref), err
        mat.close()


@pytest.mark.parametrize("n,angles", [(140, 97), (138, 98), (141, 98)])
def test_batched_groups_of_large_matrices(A, ctx, n, angles):
    # row blocks around the line of the group rule (4864 blocks of four rows),
    # whose sums do not depend on the batch's width either
    geom = W.Geometry(n, angles, 201)
    Amat = W.siddon_matrix(geom)
    mat = A.Matrix(ctx, Amat, n, angles)
    sls = [W.make_slice(Amat, geom, 300.0 * n * (1 + i % 5), W.seed_for(3, i), phantom="uniform")
           for i in range(66)]

    def run(K):
        g = torch.from_numpy(np.stack([s.g for s in sls[:K]])).to(DEV)
        gam = torch.from_numpy(np.stack([s.gamma for s in sls[:K]])).to(DEV)
        f = torch.empty((K, mat.d), dtype=torch.float32, device=DEV)
        A.appga_reconstruct_batched(ctx.handle, mat.handle, K, g, gam, None,
                                    A.default_params(**PAR), f)
        return f.cpu().numpy()

    whole = run(66)
    for K in (1, 9, 17, 33):
        np.testing.assert_array_equal(run(K), whole[:K])
    for i in (0, 65):
        ref = O.appga(O.Problem(Amat, sls[i].g, sls[i].gamma, n), O.Params(**PAR),
                      n_angles=angles, track_phi=False).f
        assert np.linalg.norm(whole[i] - ref) <= 5e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,angles,bins", [(16, 10, 8), (178, 6, 253), (247, 5, 350),
                                           (24, 3734, 34), (24, 7484, 34)])
def test_single_projections_touch_only_their_entries(A, ctx, n, angles, bins):
    # entries a row does not have are never read into it: an infinite vector
    # entry reaches exactly the rows that hold it, an empty row stays zero, and
    # the other rows keep the accuracy of double-float / compensated sums
    geom = W.Geometry(n, angles, bins)
    Amat = W.siddon_matrix(geom).astype(np.float64)
    mat = A.Matrix(ctx, Amat.astype(np.float32), n, angles)
    m, d = Amat.shape
    rng = np.random.default_rng(2)
    f = rng.random(d).astype(np.float32)
    w = rng.standard_normal(m).astype(np.float32)
    y_ref, b_ref = Amat @ f, Amat.T @ w
    hit = np.asarray(Amat.sum(axis=1)).ravel() > 0
    for x in (0, d // 2 + n // 2):
        f[x] = np.inf
        w[x % m] = np.inf
        y = torch.empty(m, dtype=torch.float64, device=DEV)
        one = torch.ones(m, dtype=torch.float32, device=DEV)
        A.appga_forward_ratio(ctx.handle, mat.handle, torch.from_numpy(f).to(DEV), one, one, y)
        out = torch.empty(d, dtype=torch.float32, device=DEV)
        A.appga_backproject(ctx.handle, mat.handle, torch.from_numpy(w).to(DEV), out)
        y, out = y.cpu().numpy(), out.cpu().numpy()
        col = np.zeros(m, bool)
        for xx in np.nonzero(~np.isfinite(f))[0]:
            col |= Amat[:, [xx]].toarray().ravel() != 0
        row = np.zeros(d, bool)
        for xx in np.nonzero(~np.isfinite(w))[0]:
            row |= Amat[[xx]].toarray().ravel() != 0
        assert np.all(~np.isfinite(y[col])) and np.all(y[~hit] == 0)
        assert np.all(np.abs(y - y_ref)[~col] <= 1e-11 * y_ref[~col])
        assert not np.isfinite(out[row]).any()
        bound = 3e-7 * (Amat.T @ np.where(np.isfinite(w), np.abs(w), 0))
        assert np.all(np.abs(out - b_ref)[~row] <= bound[~row])
