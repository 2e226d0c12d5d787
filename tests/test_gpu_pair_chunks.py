"""Tensor-core pairwise product: chunks whose sources share z (their z term is
formed once per chunk) and chunks that do not, against the FP64 application."""
import numpy as np
import pytest

from kl_inputs import random_block

pytestmark = pytest.mark.gpu


# (13, 3, 4) and smaller planes: chunks of 64 cross planes of equal z; (33, 9, 2):
# most lie inside one; the projective cube has none
@pytest.mark.parametrize("geometry,elems", [("cube", (13, 3, 4)), ("cube", (33, 9, 2)), ("annulus", (3, 2, 9)),
                                            ("projective_cube", (14, 5, 3)), ("cube", (65,)), ("cube", (9, 21))])
@pytest.mark.parametrize("kernel", ["gauss", "exp_sep", "exp", "matern32", "const"])
@pytest.mark.parametrize("precision,k", [("bf16", 5), ("bf16", 17), ("tf32", 3), ("tf32", 33)])
def test_against_fp64(geometry, elems, kernel, precision, k):
    import torch
    import paper_2101_00629_gb300 as kl
    out = []
    for prec in ("fp64", precision):
        geo = (0.5, 0.25, -0.2) if geometry == "projective_cube" else (1.0, 2.0, 1.0)
        h = kl.kl_create(kl.params(geometry=geometry, degree=2, elems=elems, kernel=kernel, L=0.7, geo=geo,
                                   method="collocation", precision=prec, block_k=k), torch.cuda.current_stream())
        try:
            N, _, _ = kl.kl_dims(h)
            X = torch.from_numpy(random_block(N, k, 3)).cuda()
            Y = [torch.empty_like(X) for _ in range(2)]
            for y in Y:
                kl.kl_apply_A(h, X, N, y, N, k)
            torch.cuda.synchronize()
            assert torch.equal(Y[0], Y[1])
            out.append(Y[0].cpu().numpy())
        finally:
            kl.kl_destroy(h)
    # |x| weighted by the kernel's largest value bounds every entry's terms;
    # 5e-5 of that is the tolerance of the mixed parity tests
    scale = np.abs(out[0]).max(axis=1, keepdims=True)
    assert np.all(np.abs(out[1] - out[0]) <= 5e-5 * np.maximum(scale, 1e-3))
