"""Fields that decay along x, along y or away from a ridge: the register-tile kernels take regions in block fixed point
only where every cell keeps float64's significant bits, whichever way the field decays. Compared cell by cell with the
per-operation kernels (fas_params.path = 1), relative to the field's size at that cell; the bar is the library's for
fixed-cycle iterates. 2^-100 over the grid is 2^-25 over one region of 64 columns."""
import numpy as np
import pytest

from workloads import random_field

pytestmark = pytest.mark.gpu


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _decay(kind, shape):
    j, i = np.indices(shape)
    at = {"x": i, "y": j, "ridge": np.abs(i - 2 * j), "-x": shape[1] - 1 - i}[kind]
    return 2.0 ** (-100.0 * at / 256.0)


# coarse cells stay small against the decay where the field falls on both axes: a correction is constant over a coarse
# cell, and float64 itself loses what the field falls over one (2^-24 on a ridge over 128 x 128 cells down to 4 x 4)
CASES = [(shape, 4, kind) for shape in ((128, 256), (256, 256), (32, 32)) for kind in ("x", "-x", "y")] + \
        [((128, 128), 32, "ridge"), ((64, 64), 4, "ridge"), ((32, 32), 4, "ridge")]


@pytest.mark.parametrize("varying", [False, True])
@pytest.mark.parametrize("shape,coarsest,kind", CASES)
def test_decaying_fields(cuda_lib, shape, coarsest, kind, varying):
    fas = cuda_lib
    D = _decay(kind, shape)
    u0, f = D * random_field(shape, 701, 1, 2), D * random_field(shape, 702, 1, 2)
    kappa = _t(random_field(shape, 703, 0.5, 1.5)) if varying else None
    out = []
    for path in (0, 1):
        ctx = fas.fas_create(fas.make_params(shape, 1.0 / 256, beta=2e-5, path=path, coarsest=coarsest), kappa=kappa)
        u, ft = _t(u0), _t(f)
        for _ in range(3):
            fas.fas_vcycle(ctx, u, ft)
        out.append(u.cpu().numpy())
    assert np.max(np.abs(out[0] - out[1]) / (D + np.abs(out[1]))) <= 1e-12
