"""The residual norm of float64 2D solves (fas_info.res0, res) against the norm of the residual formed here from
the fields themselves, in extended precision.

The kernels hold a cell's scaled residual as an integer: one unit is at most 2^-55 of the largest |u| of its region
(V(2,2)), times the diagonal d for the residual itself. The grids' h and the coefficients are powers of two (or
few-bit numbers), so the operator has no rounding of its own."""
import numpy as np
import pytest

from oracle import cell_centred as cc
from workloads import noisy_cos_mode, normal, random_field

pytestmark = pytest.mark.gpu

N_, D_ = cc.NEUMANN, cc.DIRICHLET


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _operator(shape, h, bc, kappa=1.0):
    kappa = kappa if np.isscalar(kappa) else np.asarray(kappa, dtype=np.longdouble)
    return cc.Operator(shape, h, 1.0, 1.0, kappa, bc, dtype=np.longdouble)


def _norm(r):
    return float(np.sqrt(np.sum(r * r)))


def _few_bits(shape, seed):
    return 0.5 + np.floor(16.0 * random_field(shape, seed)) / 16.0


@pytest.mark.parametrize("signs", ["both", "negative", "positive"])
@pytest.mark.parametrize("k", [34, 100, 1000])
@pytest.mark.parametrize("varying", [False, True])
def test_residual_norm_of_a_few_units(cuda_lib, varying, k, signs):
    """Residuals with an rms of k units, of both signs or of one. Forming one costs at most about one unit (three
    roundings of half a unit); with a per-cell diffusivity also the weights' float64 rounding, some 4 units: the
    norm is off by at most (4^2 / k^2) of itself there, and by half a unit of k where all have one sign."""
    fas = cuda_lib
    shape, h = (512, 512), 1.0 / 512
    kappa = _few_bits(shape, 672) if varying else 1.0
    op = _operator(shape, h, (N_,) * 4, kappa)
    u = 1.5 + 0.25 * noisy_cos_mode(shape, 671, 0.0)
    d = 4.0 / (h * h)
    unit = d * 2.0 ** -55 * float(np.max(np.abs(u)))
    noise = normal(673, 1, u.size).reshape(shape)
    noise = {"both": noise, "negative": -np.abs(noise), "positive": np.abs(noise)}[signs]
    f = np.asarray(cc.apply_A(op, u) + k * unit * noise, dtype=np.float64)
    true = _norm(cc.residual(op, u, f))
    ctx = fas.fas_create(fas.make_params(shape, h), kappa=_t(kappa) if varying else None)
    info = fas.fas_vcycle(ctx, _t(u), _t(f))
    assert abs(info.res0 - true) <= (0.5 / k + (16.0 if varying else 1.0) / k ** 2) * true


def test_solves_of_f_and_minus_f(cuda_lib):
    """The residuals at the stopping test are some 50 units here. The roundings of the two runs differ, by up to a
    unit a cell: 1e-5 of the norm of 2^20 cells."""
    fas = cuda_lib
    shape, h, bc = (1024, 1024), 1.0 / 1024, (D_,) * 4
    f = 10.0 * noisy_cos_mode(shape, 681, 0.3)
    infos, us = [], []
    for s in (1.0, -1.0):
        ctx = fas.fas_create(fas.make_params(shape, h, bc=bc, kmax=60))
        u = _t(0 * f)
        infos.append(fas.fas_solve(ctx, u, _t(s * f)))
        us.append(u.cpu().numpy())
    assert infos[0].cycles == infos[1].cycles
    assert abs(infos[0].res - infos[1].res) <= 1e-4 * infos[0].res
    true = _norm(cc.residual(_operator(shape, h, bc), us[0], f))
    assert abs(infos[0].res - true) <= 1e-2 * true
