"""3D float64 V-cycles through the default path (small levels restricted with the residuals of a coarse cell spread
over lanes) against the reference path (one coarse cell per thread), cells and faces. Both sides round differently, a
few units of 2^-53 per operation: the bar is the library's for fixed-cycle iterates."""
import numpy as np
import pytest

from oracle import cell_centred as cc
from workloads import noisy_cos_mode, random_field, zero_wall_slot

pytestmark = pytest.mark.gpu

N_, D_, P_ = cc.NEUMANN, cc.DIRICHLET, cc.PERIODIC


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("shape,bc,fax", [
    ((8, 8, 8), (N_,) * 6, None), ((16, 32, 8), (D_,) * 6, None), ((32, 16, 64), (P_,) * 6, None),
    ((64, 32, 32), (N_, D_, P_, P_, D_, D_), None), ((4, 64, 256), (N_,) * 6, None),
    ((16, 16, 16), (D_,) * 6, 0), ((32, 16, 8), (D_,) * 6, 1), ((16, 64, 32), (D_,) * 6, 2)])
def test_small_levels(cuda_lib, shape, bc, fax):
    fas = cuda_lib
    u0, f = random_field(shape, 751, -1, 1), noisy_cos_mode(shape, 752)
    kw = {}
    if fax is not None:
        kw["location"] = fas.FAS_FACE_X + fax
        u0, f = zero_wall_slot(u0, fax), zero_wall_slot(f, fax)
    out = []
    for path in (0, 1):
        ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=2e-3, bc=bc, coarsest=2, path=path, **kw))
        u, ft = _t(u0), _t(f)
        for _ in range(3):
            fas.fas_vcycle(ctx, u, ft)
        out.append(u.cpu().numpy())
    assert np.max(np.abs(out[0] - out[1])) <= 1e-12 * np.max(np.abs(out[1]))
