"""Operations that sum the neighbours of several cells at one integer scale, on fields that differ by 2^20 from one
cell to the next: each cell keeps the accuracy of float64 arithmetic on its own stencil."""
import numpy as np
import pytest

from oracle import cell_centred as cc
from oracle import staggered as st
from workloads import random_field, zero_wall_slot

pytestmark = pytest.mark.gpu

N_, D_, P_ = cc.NEUMANN, cc.DIRICHLET, cc.PERIODIC
EPS = 2.0 ** -53


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _steep(shape, seed, lo=1.0):
    i = np.indices(shape)[-1]
    step = np.minimum(i % 16, 16 - i % 16)  # 2^0 .. 2^-160 and back along x
    return 2.0 ** (-20.0 * step) * random_field(shape, seed, lo, 2)


CASES = [((32, 64), (N_,) * 4, None), ((64, 128), (D_, N_, P_, P_), None), ((64, 64), (D_,) * 4, 0),
         ((16, 32, 64), (N_,) * 6, None), ((16, 16, 32), (P_, P_, D_, N_, N_, N_), None), ((16, 16, 32), (D_,) * 6, 0),
         ((16, 16, 32), (D_,) * 6, 2)]


@pytest.mark.parametrize("shape,bc,fax", CASES)
@pytest.mark.parametrize("ir", [False, True])
def test_residual_keeps_small_cells(cuda_lib, ir, shape, bc, fax):
    """fas_residual and the refinement residual: within 16 roundings of 2^-53 of the sum of the stencil's terms (and
    the rounding to float32)."""
    import torch
    fas = cuda_lib
    h, beta = 1.0 / 64, 2.0 ** -10
    u, f = _steep(shape, 711, -2), _steep(shape, 712, -2)
    kw = {}
    if fax is None:
        op = cc.Operator(shape, h, 1.0, beta, 1.0, bc, dtype=np.longdouble)
        exact = cc.residual(op, u, f)
    else:
        u = zero_wall_slot(u, fax)
        kw["location"] = fas.FAS_FACE_X + fax
        op = st.FaceOperator(shape, h, 1.0, beta, fax, dtype=np.longdouble)
        exact = st.residual_face(op, u, f)
    # sum of the magnitudes of a cell's terms: neighbours (wrapped or not: an upper bound) and diagonal
    c = beta / (h * h)
    scale = np.abs(f) + (1.0 + 4 * len(shape) * c) * np.abs(u)
    for ax in range(len(shape)):
        for s in (-1, 1):
            scale = scale + c * np.abs(np.roll(u, s, ax))
    ctx = fas.fas_create(fas.make_params(shape, h, beta=beta, bc=bc, **kw))
    if ir:
        out = torch.empty(u.size, dtype=torch.float32, device="cuda")
        fas.fas_residual_ir(ctx, _t(u), _t(f), out)
    else:
        out = torch.empty(u.size, dtype=torch.float64, device="cuda")
        fas.fas_residual(ctx, 0, _t(u), _t(f), out)
    got = out.cpu().numpy().astype(np.float64).reshape(shape)
    tiny = 2.0 ** -149 if ir else 0.0
    bar = 16 * EPS * scale + (2.0 ** -24 * np.abs(exact) if ir else 0.0) + tiny
    assert np.max(np.abs(got - exact) / bar) <= 1.0


@pytest.mark.parametrize("shape,bc", [(s, b) for s, b, fx in CASES if fx is None])
def test_smoothing_keeps_small_cells(cuda_lib, shape, bc):
    """One sweep on positive data: every update is a sum of positive terms (at most seven roundings each, and those
    of the first colour's values)."""
    fas = cuda_lib
    h, beta = 1.0 / 64, 2.0 ** -10
    u, f = _steep(shape, 721), _steep(shape, 722)
    op = cc.Operator(shape, h, 1.0, beta, 1.0, bc, dtype=np.longdouble)
    want = np.array(u, dtype=np.longdouble)
    cc.xmcgs_sweep(op, want, f)
    ctx = fas.fas_create(fas.make_params(shape, h, beta=beta, bc=bc))
    ut = _t(u)
    fas.fas_smooth(ctx, 0, ut, _t(f), 1)
    assert np.max(np.abs(ut.cpu().numpy() - want) / want) <= 24 * EPS
