"""Norms formed by one block, by a few and by a full grid of blocks. Every value is rounded to float32 before it is squared
and every square once more: the norm is within 2^-23 of the exact one whatever the number of cells a thread adds up."""
import numpy as np
import pytest

from workloads import random_field

pytestmark = pytest.mark.gpu

N_ = 0


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("varying", [False, True])
@pytest.mark.parametrize("shape", [(4, 4), (16, 16), (32, 32), (64, 64), (256, 512), (1024, 512), (4096, 2048), (4, 4, 4),
                                   (8, 8, 8), (8, 16, 16), (64, 64, 32), (128, 128, 128)])
def test_norms(cuda_lib, shape, varying):
    import torch
    fas = cuda_lib
    u, f = random_field(shape, 771, -1, 1), random_field(shape, 772, -1, 1)
    kappa = _t(random_field(shape, 773, 0.5, 1.5)) if varying else None
    ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=1e-3, precision=1, use_graph=0), kappa=kappa)
    ut, ft = _t(u), _t(f)
    r = torch.empty_like(ut)
    r32 = torch.empty(u.size, dtype=torch.float32, device="cuda")
    for norm, field in ((fas.fas_residual(ctx, 0, ut, ft, r), r), (fas.fas_residual_ir(ctx, ut, ft, r32), r32)):
        exact = float(torch.linalg.vector_norm(field.double()))
        assert abs(norm - exact) <= 2.0 ** -23 * exact
    info = fas.fas_vcycle(ctx, ut, ft)
    assert abs(info.res0 - float(torch.linalg.vector_norm(r.double()))) <= 2.0 ** -20 * info.res0
