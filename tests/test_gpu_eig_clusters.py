"""The small non-symmetric eigensolver on clusters of equal eigenvalues that
rounding or a coarse operator has split by 1e-10 (a cube's threefold K-L
eigenvalues): its Schur form is a backward-stable one of the given matrix, in
FP64 with FP64's tolerance."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FP64, DOUBLE_FLOAT = 0, 2


def _solve(H, arith):
    import torch
    import paper_2101_00629_gb300 as kl
    lib = ctypes.CDLL(kl.library_path())
    # kl::launch_nonsym_eig and kl::nonsym_eig_work_doubles (csrc/kl_internal.h)
    eig = getattr(lib, "_ZN2kl17launch_nonsym_eigEPKdiPdS2_S2_S2_S2_PiP11CUstream_stii")
    size = getattr(lib, "_ZN2kl23nonsym_eig_work_doublesEi")
    size.restype = ctypes.c_int64
    n = H.shape[0]
    d = [torch.from_numpy(np.ascontiguousarray(H.T)).cuda()]
    d += [torch.zeros(m, dtype=torch.float64, device="cuda") for m in (n, n, n * (n + 1), n * n, size(n))]
    status = torch.full((4,), -1, dtype=torch.int32, device="cuda")
    p = [ctypes.c_void_p(t.data_ptr()) for t in d + [status]]
    rc = eig(p[0], n, *p[1:], ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), n, arith)
    torch.cuda.synchronize()
    assert rc == 0
    return int(status[0]), d[2].cpu().numpy(), d[4].cpu().numpy().reshape(n, n).T


@pytest.mark.parametrize("arith,eps", [(FP64, 2.0 ** -52), (DOUBLE_FLOAT, 1e-13)])
@pytest.mark.parametrize("n", [12, 24, 48, 96, 201])
@pytest.mark.parametrize("split", [3e-10, 1e-12, 0.0])
def test_threefold_eigenvalues(n, split, arith, eps):
    rng = np.random.default_rng(1000 * n + 1)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.repeat(0.7 ** np.arange(n // 3), 3)
    H = Q @ np.diag(lam) @ Q.T + split * rng.standard_normal((n, n)) / np.sqrt(n)
    status, wi, Z = _solve(H, arith)
    assert status == 0
    F = np.linalg.norm(H)
    # a backward-stable decomposition: about 2 n steps of n reflectors each
    # leave 10 n eps ||H||_F, and a deflation drops an entry of n eps ||H||
    tol = 11 * n * eps
    assert np.abs(Z.T @ Z - np.eye(n)).max() <= tol
    T = Z.T @ H @ Z
    # quasi-triangular: below the diagonal only the 2 x 2 blocks of complex
    # pairs, which no other row touches
    low = np.abs(np.tril(T, -1))
    pair = np.flatnonzero(wi[:-1] > 0)
    low[pair + 1, pair] = 0.0
    assert low.max() <= tol * F
