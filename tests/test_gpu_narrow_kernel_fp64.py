"""An FP64 collocation solve whose projected matrices hold clusters at the
operator's rounding (narrow Gaussian, many wanted pairs): the small FP64
eigensolver does not converge for this start block and the double-float one
takes over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,seed", [(8, 7)])
def test_narrow_gaussian_collocation(k, seed):
    import torch
    import paper_2101_00629_gb300 as kl
    M = 62
    h = kl.kl_create(kl.params(geometry="cube", degree=3, elems=(8, 8, 8), kernel="gauss", L=0.12838993824229705,
                               method="collocation", precision="fp64", block_k=k, seed=seed),
                     torch.cuda.current_stream())
    try:
        lam, res = np.zeros(M), np.zeros(M)
        rc = kl.kl_eigs(h, M, 1e-8, lam, None, 0, 0, res)
        assert rc in (kl.KL_OK, kl.KL_WARN_COMPLEX)
        assert np.all(np.isfinite(lam)) and np.all(np.diff(lam) <= 1e-12 * lam[0]) and res.max() <= 1e-8
    finally:
        kl.kl_destroy(h)
