"""The column-streaming 3D float32 kernels on levels that they take (at least 2^21 cells), bit for bit against the
per-operation kernels: one and two sweeps, every boundary kind, grids narrower than a region of 64 columns x 64 rows,
few planes, and two column levels (the coarser one with the tau correction). The number of launches shows that they ran."""
import numpy as np
import pytest

from workloads import noisy_cos_mode, random_field

pytestmark = pytest.mark.gpu

N_, D_, P_ = 0, 1, 2
MIXED_BC = (N_, D_, D_, N_, N_, D_)


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("shape,bc,nu,inner", [
    ((128, 128, 128), (N_,) * 6, 1, 2), ((128, 128, 128), (D_,) * 6, 2, 2), ((128, 128, 128), (P_,) * 6, 1, 2),
    ((64, 256, 128), (P_, P_, N_, D_, P_, P_), 2, 2), ((256, 64, 128), (N_, N_, P_, P_, D_, D_), 2, 1),
    ((64, 64, 512), MIXED_BC, 1, 2), ((512, 64, 64), (D_,) * 6, 2, 2), ((512, 64, 64), (P_,) * 6, 2, 1),
    ((32, 512, 128), (N_, N_, N_, N_, P_, P_), 1, 1),
    # two levels of the column kernels
    ((256, 256, 256), (D_,) * 6, 1, 1), ((256, 256, 256), (P_,) * 6, 2, 2), ((512, 128, 256), MIXED_BC, 2, 2),
    ((128, 512, 256), (P_, P_, D_, N_, N_, N_), 1, 2)])
def test_column_levels_match_per_operation(cuda_lib, shape, bc, nu, inner):
    fas = cuda_lib
    u0, f = random_field(shape, 731, -1, 1), noisy_cos_mode(shape, 732)
    out, launches = [], []
    for path in (0, 1):
        ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=2e-3, bc=bc, nu1=nu, nu2=nu, precision=1,
                                             inner_cycles=inner, path=path))
        u, ft = _t(u0), _t(f)
        for _ in range(2):
            fas.fas_vcycle(ctx, u, ft)
        out.append(u.cpu().numpy())
        launches.append(fas.fas_launch_count(ctx))
        fas.fas_destroy(ctx)
    np.testing.assert_array_equal(out[0], out[1])
    # a level in two launches instead of at least 4 nu + 2
    assert launches[0] <= launches[1] - 2 * inner * (4 * nu - 1)
