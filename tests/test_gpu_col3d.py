"""The column-streaming 3D float32 kernels (mixed precision, fas_params.path 0) against the per-operation
kernels (path 1), bit for bit, at sizes around one region (64 columns x 64 rows, segments of planes), thin
grids, every boundary kind, one and two sweeps, one to three float32 cycles per step."""
import numpy as np
import pytest

from workloads import noisy_cos_mode, random_field

pytestmark = pytest.mark.gpu

N_, D_, P_ = 0, 1, 2


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("shape,bc,nu,inner", [
    ((32, 32, 32), (N_,) * 6, 2, 1), ((64, 64, 64), (D_, N_, N_, D_, D_, N_), 2, 2), ((128, 64, 128), (D_,) * 6, 2, 2),
    ((16, 128, 256), (N_,) * 6, 1, 2), ((256, 32, 16), (N_, D_, N_, N_, N_, N_), 2, 2),
    ((64, 32, 128), (P_,) * 6, 2, 2), ((32, 128, 64), (P_, P_, N_, D_, P_, P_), 1, 3),
    ((128, 128, 32), (N_, N_, P_, P_, D_, D_), 2, 1), ((128, 256, 256), (N_,) * 6, 2, 2)])
def test_column_kernels_match_per_operation(cuda_lib, shape, bc, nu, inner):
    fas = cuda_lib
    u0, f = random_field(shape, 641, -1, 1), noisy_cos_mode(shape, 642)
    out = []
    for path in (0, 1):
        ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=2e-3, bc=bc, nu1=nu, nu2=nu, precision=1,
                                             inner_cycles=inner, path=path))
        u, ft = _t(u0), _t(f)
        for _ in range(2):
            fas.fas_vcycle(ctx, u, ft)
        out.append(u.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
