"""Banded mass and collocation solves along the directions (GPU) against dense
1D solves of the oracle's matrices, at the sizes where blocks of lines, the
shared-memory limit and the choice of the dense product end."""
import numpy as np
import pytest

from kl_inputs import random_block
from oracle import splines
from oracle.problem import Problem

pytestmark = pytest.mark.gpu


def _one_d(prob, method, d):
    t = prob.trial_knots()[d]
    if method == "collocation":
        return splines.bspline_basis(t, prob.p, splines.greville(t, prob.p))
    x, w = splines.element_gauss(t, prob.p + 1)
    B = splines.bspline_basis(t, prob.p, x)
    return B.T @ (w[:, None] * B)


@pytest.mark.parametrize("method", ["galerkin", "collocation"])
@pytest.mark.parametrize("p,elems,k", [
    (1, (5, 4, 3), 1),           # dense: too little work for the sweeps
    (2, (300,), 3),
    (1, (29, 14, 23), 37),       # banded sweeps from here on
    (2, (70, 33), 130),          # two directions
    (2, (31, 17, 9), 64),
    (3, (64, 3, 2), 256),        # 67 x 6 x 5: ragged blocks of lines
    (2, (130, 2, 3), 200),
    (2, (550, 1), 256),          # 552 points, the most that fit
    (2, (551, 1), 256),          # 553: dense
    (2, (62, 40, 12), 33),       # blocks of 64 lines
    (8, (42, 21, 10), 90),
    (6, (13, 40, 14), 40),
])
def test_zinv(method, p, elems, k):
    import torch
    import paper_2101_00629_gb300 as kl
    prob = Problem("cube", p, elems, "gauss", 1.0, 0.5)
    h = kl.kl_create(kl.params(geometry="cube", degree=p, elems=elems, method=method), torch.cuda.current_stream())
    try:
        N, _, _ = kl.kl_dims(h)
        X = random_block(N, k, 5)
        Xd = torch.from_numpy(X).cuda()
        Y = torch.empty_like(Xd)
        kl.kl_apply_Zinv(h, Xd, N, Y, N, k)
        kl.kl_apply_Zinv(h, Xd, N, Xd, N, k)  # in place
        assert torch.equal(Xd, Y)
        n = [e + p for e in elems] + [1] * (3 - len(elems))
        Z = [_one_d(prob, method, d) for d in range(len(elems))] + [np.eye(1)] * (3 - len(elems))
        got = Y.cpu().numpy().reshape(k, n[2], n[1], n[0])
        # residual: a backward-stable solve leaves |Z y - x| at a few n eps |Z||y|
        res, mag = got, np.abs(got)
        for d, sub in enumerate(("ai,zkji->zkja", "aj,zkji->zkai", "ak,zkji->zaji")):
            res = np.einsum(sub, Z[d], res)
            mag = np.einsum(sub, np.abs(Z[d]), mag)
        err = np.abs(res - X.reshape(res.shape))
        cond = np.prod([np.linalg.norm(np.linalg.inv(z) @ np.abs(z), np.inf) for z in Z])
        assert np.all(err <= 64 * sum(n) * 2.0 ** -53 * cond * np.abs(mag).max(axis=(1, 2, 3), keepdims=True))
    finally:
        kl.kl_destroy(h)


@pytest.mark.parametrize("geometry,p,elems,method", [
    ("cube", 2, (20, 9, 14), "galerkin"),
    ("half_annulus", 2, (24, 5, 13), "galerkin"),
    ("annulus", 3, (12, 7, 9), "galerkin"),
    ("cube", 2, (17, 3, 12), "galerkin_std"),
])
def test_standard_form_as_solves(geometry, p, elems, method):
    """A' of a wide block (banded solves around banded tables) against the same
    columns one at a time (dense tables)."""
    import torch
    import paper_2101_00629_gb300 as kl
    k = 64
    h = kl.kl_create(kl.params(geometry=geometry, degree=p, elems=elems, kernel="exp", L=0.8, method=method, block_k=k),
                     torch.cuda.current_stream())
    try:
        N, _, _ = kl.kl_dims(h)
        Xd = torch.from_numpy(random_block(N, k, 9)).cuda()
        Y, Z = torch.empty_like(Xd), torch.empty_like(Xd)
        kl.kl_apply_Aprime(h, Xd, N, Y, N, k)
        for c in range(0, k, 21):
            kl.kl_apply_Aprime(h, Xd[c], N, Z[c], N, 1)
            err = (Y[c] - Z[c]).norm() / Z[c].norm()
            assert err <= 1e-12, (c, err)
    finally:
        kl.kl_destroy(h)


@pytest.mark.parametrize("ldx,ldy,shift", [(0, 5, 0), (5, 0, 0), (0, 0, 7), (3, 0, -11)])
@pytest.mark.parametrize("method", ["galerkin", "collocation"])
def test_zinv_overlapping_blocks(method, ldx, ldy, shift):
    """X and Y in one buffer with different leading dimensions or offsets."""
    import torch
    import paper_2101_00629_gb300 as kl
    k = 64
    h = kl.kl_create(kl.params(geometry="cube", degree=2, elems=(31, 17, 9), kernel="gauss", L=0.5, method=method),
                     torch.cuda.current_stream())
    try:
        N, _, _ = kl.kl_dims(h)
        X = torch.from_numpy(random_block(N, k, 3)).cuda()
        Y = torch.empty_like(X)
        kl.kl_apply_Zinv(h, X, N, Y, N, k)
        buf = torch.zeros(k * (N + 16) + 64, dtype=torch.float64, device="cuda")
        x = buf[32:].as_strided((k, N), (N + ldx, 1))
        y = buf[32 + shift:].as_strided((k, N), (N + ldy, 1))
        x.copy_(X)
        kl.kl_apply_Zinv(h, x, N + ldx, y, N + ldy, k)
        assert torch.equal(y, Y)
    finally:
        kl.kl_destroy(h)


@pytest.mark.parametrize("apply", ["Zinv", "Aprime"])
@pytest.mark.parametrize("geometry,p,geo", [
    ("projective_cube", 2, (0.5, 0.25, -0.2)),  # weights before and after the sweeps
    ("projective_cube", 3, (-0.4, 0.3, 0.6)),
    ("half_annulus", 2, (1.0, 2.0, 1.0)),       # Greville points of joined knots
    ("half_annulus", 3, (1.0, 2.0, 1.0)),
])
def test_collocation_sweeps(geometry, p, geo, apply):
    """Z^-1 and A' of a wide block (banded sweeps) against the same columns one
    at a time (dense inverses)."""
    import torch
    import paper_2101_00629_gb300 as kl
    k, elems = 64, (20, 14, 16)
    h = kl.kl_create(kl.params(geometry=geometry, degree=p, elems=elems, kernel="gauss", L=0.8, method="collocation",
                               precision="fp64", geo=geo), torch.cuda.current_stream())
    try:
        N, _, _ = kl.kl_dims(h)
        call = kl.kl_apply_Zinv if apply == "Zinv" else kl.kl_apply_Aprime
        X = torch.from_numpy(random_block(N, k, 13)).cuda()
        Y, Y1 = torch.empty_like(X), torch.empty_like(X)
        call(h, X, N, Y, N, k)
        Z = [_one_d(Problem(geometry, p, elems, "gauss", 1.0, 0.8, geo=geo), "collocation", d) for d in range(3)]
        cond = np.prod([np.linalg.norm(np.abs(np.linalg.inv(z)) @ np.abs(z), np.inf) for z in Z])
        # two backward-stable solves by direction (at most 2 n units each), and
        # for A' two pairwise products in other column blocks (1e-13)
        tol = 8 * sum(z.shape[0] for z in Z) * cond * 2.0 ** -53 + (1e-13 * cond if apply == "Aprime" else 0.0)
        for c in range(0, k, 21):
            call(h, X[c], N, Y1[c], N, 1)
            err = float((Y[c] - Y1[c]).abs().max() / Y1[c].abs().max())
            assert err <= tol, (c, err, tol)
    finally:
        kl.kl_destroy(h)
