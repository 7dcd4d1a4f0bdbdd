"""The fused Arnoldi steps (one cooperative launch per 16 steps) against the
dense solution and the oracle: block widths at the kernel's instances (4 and 16
columns), more columns than it takes, sizes below a warp, runs that end inside
a batch and restarts shorter than one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_01464_gb300 import qpinv
    c = qpinv.Context(0)
    yield c
    c.close()


def _system(n, m, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((4, n, n)) / np.sqrt(4 * n) / 4
    A[0] += np.eye(n)
    return A, rng.standard_normal((4, n, m))


@pytest.mark.parametrize("n,m", [(1, 1), (5, 2), (31, 4), (33, 5), (100, 16), (64, 17), (150, 3)])
@pytest.mark.parametrize("kind", ["gmres", "fom"])
@pytest.mark.parametrize("restart", [0, 7])
def test_krylov_solution(ctx, n, m, kind, restart):
    # kappa(A) < 2: a residual of 1e-11 bounds the error by 2e-11 of the solution
    A, B = _system(n, m, 10 * n + m)
    X, info = ctx.global_krylov(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), kind, restart=restart,
                                tol=1e-11, max_iter=400)
    from paper_2605_01464_gb300 import inputs
    ref = inputs.unchi(np.linalg.solve(inputs.chi(A), inputs.chi(B)))
    assert info["converged"]
    assert np.linalg.norm(X.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (7, 15, 9), (8, 16, 8), (9, 17, 17), (250, 33, 70)])
def test_fp64_product_tiles(ctx, m, k, n):
    import oracle
    rng = np.random.default_rng(m + k + n)
    A, B = rng.standard_normal((4, m, k)), rng.standard_normal((4, k, n))
    C = ctx.qgemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), precision="fp64").cpu().numpy()
    # 4 k products summed in FP64, in both
    tol = 8 * k * 2.0 ** -53 * (np.linalg.norm(A, axis=(0, 2))[:, None] * np.linalg.norm(B, axis=(0, 1))[None])
    assert np.all(np.abs(C - oracle.matmul(A, B)) <= tol)
