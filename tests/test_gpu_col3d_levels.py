"""The column-streaming 3D float32 kernels on levels that they take (at least 2^24 cells), bit for bit against the
per-operation kernels: one and two sweeps, every boundary kind, grids narrower than a region of 64 columns x 64 rows,
few planes, and two column levels (the coarser one with the tau correction). The number of launches shows that they ran."""
import pytest

pytestmark = pytest.mark.gpu

N_, D_, P_ = 0, 1, 2
MIXED_BC = (N_, D_, D_, N_, N_, D_)


@pytest.mark.parametrize("shape,bc,nu,inner", [
    ((256, 256, 256), (N_,) * 6, 1, 2), ((256, 256, 256), (D_,) * 6, 2, 2), ((256, 256, 256), (P_,) * 6, 1, 2),
    ((128, 512, 256), (P_, P_, N_, D_, P_, P_), 2, 2), ((512, 256, 128), (N_, N_, P_, P_, D_, D_), 2, 1),
    ((64, 512, 512), MIXED_BC, 1, 2), ((1024, 512, 64), (D_,) * 6, 2, 2), ((1024, 256, 64), (P_,) * 6, 2, 1),
    ((2048, 256, 32), (N_,) * 6, 2, 2), ((2048, 32, 256), (N_, N_, P_, P_, D_, D_), 2, 1),
    ((64, 1024, 256), (N_, N_, N_, N_, P_, P_), 1, 1),
    # two levels of the column kernels
    ((512, 512, 512), (D_,) * 6, 1, 1), ((256, 1024, 512), (P_,) * 6, 2, 2), ((1024, 256, 512), MIXED_BC, 2, 2),
    ((512, 512, 512), (P_, P_, D_, N_, N_, N_), 1, 2)])
def test_column_levels_match_per_operation(cuda_lib, shape, bc, nu, inner):
    import torch
    fas = cuda_lib
    gen = torch.Generator("cuda").manual_seed(731)
    u0 = 2.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    f = torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen)
    out, launches = [], []
    for path in (0, 1):
        ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=2e-3, bc=bc, nu1=nu, nu2=nu, precision=1,
                                             inner_cycles=inner, path=path, coarsest=2))
        u = u0.clone()
        for _ in range(2):
            fas.fas_vcycle(ctx, u, f)
        out.append(u)
        launches.append(fas.fas_launch_count(ctx))
        fas.fas_destroy(ctx)
    assert torch.equal(out[0], out[1])
    # a level in two launches instead of at least 4 nu + 2
    assert launches[0] <= launches[1] - 2 * inner * (4 * nu - 1)
