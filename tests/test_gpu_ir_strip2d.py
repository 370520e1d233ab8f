"""The 2D strip kernel of the refinement residual (grids of more than 2^22 cells): r32 against exact rational
arithmetic on sampled cells, bit for bit wherever the row of 128 cells qualifies, and the same at every call."""
from fractions import Fraction

import numpy as np
import pytest

from workloads import noisy_cos_mode, random_field, uniform

pytestmark = pytest.mark.gpu

N_, D_ = 0, 1


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("bc", [(N_,) * 4, (D_, N_, N_, D_)])
@pytest.mark.parametrize("shift,cover", [(1.5, 0.95), (0.0, 0.0)])
def test_strip_residual(cuda_lib, shift, cover, bc):
    """shift 1.5: one sign, values within 2^5 of one another, so every row is exact; 0: a field that crosses zero."""
    import torch
    fas = cuda_lib
    shape = (2048, 4096)
    ny, nx = shape
    h, alpha, beta = 1.0 / 4096, 1.0, 1e-4
    u = noisy_cos_mode(shape, 741) + shift
    f = u + 1e-3 * random_field(shape, 742, -1, 1)
    ctx = fas.fas_create(fas.make_params(shape, h, alpha=alpha, beta=beta, bc=bc, precision=fas.FAS_MIXED))
    ut, ft = _t(u), _t(f)
    r32 = torch.empty(u.size, dtype=torch.float32, device="cuda")
    nrm = fas.fas_residual_ir(ctx, ut, ft, r32)
    first = r32.clone()
    for _ in range(3):
        fas.fas_residual_ir(ctx, ut, ft, r32)
        assert torch.equal(r32, first)
    got = first.cpu().numpy().reshape(shape)
    assert abs(nrm - float(np.linalg.norm(got.astype(np.float64)))) <= 1e-5 * nrm
    c = beta / (h * h)
    cells = (uniform(743, 1, 3000) * u.size).astype(np.int64)
    edge = (uniform(744, 1, 200) * nx).astype(np.int64)
    cells = np.unique(np.concatenate([cells, edge, u.size - 1 - edge, np.arange(0, u.size, nx * 16),
                                      np.arange(nx - 1, u.size, nx * 16)]))
    exact = 0
    for lin in cells:
        j, i = divmod(int(lin), nx)
        S, M = Fraction(0), 0
        for (jj, ii), face in (((j, i - 1), 0), ((j, i + 1), 1), ((j - 1, i), 2), ((j + 1, i), 3)):
            if 0 <= ii < nx and 0 <= jj < ny:
                S += Fraction(float(u[jj, ii]))
                M += 1
            elif bc[face] == D_:
                M += 2
        uc = Fraction(float(u[j, i]))
        Sd = float(S - M * uc)
        T = float(Fraction(float(f[j, i])) - Fraction(alpha) * uc)
        want = float(Fraction(c) * Fraction(Sd) + Fraction(T))
        if got[j, i].view(np.uint32) == np.float32(want).view(np.uint32):
            exact += 1
        else:  # the float64 point equation
            scale = abs(float(f[j, i])) + (alpha + 8 * c) * abs(float(u[j, i])) + 4 * c * 2.0 ** -10
            assert abs(float(got[j, i]) - want) <= 2.0 ** -23 * abs(want) + 1e-14 * scale, (j, i)
    assert exact >= cover * len(cells), (exact, len(cells))
