"""fas_info.res is the residual norm of the field that the call returns, down to float64's own rounding of it."""
import numpy as np
import pytest

from oracle import cell_centred as cc
from workloads import noisy_cos_mode

pytestmark = pytest.mark.gpu

N_, D_, P_ = cc.NEUMANN, cc.DIRICHLET, cc.PERIODIC


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("shape,bc", [((512, 512), (D_,) * 4), ((256, 512), (N_, D_, N_, N_)), ((128, 128), (P_,) * 4)])
def test_norm_of_the_returned_field_at_the_floor(cuda_lib, shape, bc):
    """After many cycles the residual is that of rounding u to float64: up to four units of 2^-55 of the region's
    largest |u| per cell, times d. Evaluating it adds three roundings of up to half a unit, a variance of a quarter."""
    fas = cuda_lib
    h = 1.0 / max(shape)
    f = 10.0 * noisy_cos_mode(shape, 691, 0.3)
    ctx = fas.fas_create(fas.make_params(shape, h, bc=bc, coarse_exact=1))
    u, ft = _t(0 * f), _t(f)
    for _ in range(30):
        info = fas.fas_vcycle(ctx, u, ft)
    un = u.cpu().numpy()
    r = cc.residual(cc.Operator(shape, h, 1.0, 1.0, 1.0, bc, dtype=np.longdouble), un, f)
    true = float(np.sqrt(np.sum(r * r)))
    unit = 4.0 / (h * h) * 2.0 ** -55 * float(np.max(np.abs(un)))
    assert abs(info.res ** 2 - true ** 2) <= 0.5 * un.size * unit ** 2
    assert info.res >= 0.9 * true
