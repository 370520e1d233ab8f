"""The register-tile kernels (2D cell levels, either precision) against the per-operation kernels
(fas_params.path = 1) at the sizes where they can go wrong: grids around one region (64 columns, 32 or
64 rows), thin grids, every boundary kind, 1..4 sweeps, both orderings.

float32 (the mixed solve's cycles): bit for bit. float64: both sides round differently (block fixed
point against float64), each within a few units of 2^-53 of the largest value per operation; the bar
is the library's for fixed-cycle iterates, 1e-12 relative max-norm."""
import numpy as np
import pytest

from workloads import noisy_cos_mode, random_field

pytestmark = pytest.mark.gpu

N_, D_, P_ = 0, 1, 2


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _cycles(fas, shape, path, u0, f, cycles=3, **kw):
    ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=2e-3, path=path, **kw))
    u, ft = _t(u0), _t(f)
    for _ in range(cycles):
        try:
            fas.fas_vcycle(ctx, u, ft)
        except fas.FasError as e:
            # the stopping norm squares float32 values with a scale between 2^-120 and 2^120, so a field of
            # 2^400 has no finite norm on either path; the cycle itself is complete
            if e.status != fas.FAS_ENONFINITE or np.max(np.abs(f)) < 2.0 ** 300:
                raise
    return u.cpu().numpy()


CASES = [((128, 128), (N_,) * 4, 2, 0), ((64, 64), (D_, N_, N_, D_), 2, 0), ((4, 4), (N_,) * 4, 2, 0),
         ((8, 16), (P_, P_, P_, P_), 1, 0), ((32, 256), (D_,) * 4, 2, 1), ((256, 32), (N_, N_, P_, P_), 3, 0),
         ((64, 128), (P_, P_, N_, D_), 2, 1), ((512, 256), (P_,) * 4, 2, 0), ((256, 512), (N_, D_, D_, N_), 4, 0),
         ((1024, 512), (N_,) * 4, 1, 0)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,bc,nu,ordering", CASES)
def test_tile_kernels_match_per_operation(cuda_lib, shape, bc, nu, ordering, precision):
    u0, f = random_field(shape, 611, -1, 1), noisy_cos_mode(shape, 612)
    kw = dict(bc=bc, nu1=nu, nu2=nu, ordering=ordering, precision=precision, inner_cycles=2)
    a, b = (_cycles(cuda_lib, shape, path, u0, f, **kw) for path in (0, 1))
    if precision == 1:
        np.testing.assert_array_equal(a, b)
    else:
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))


@pytest.mark.parametrize("kind", ["zero", "rows", "tiny", "huge", "spike"])
def test_tile_float64_scales(cuda_lib, kind):
    """Fields whose regions fixed point cannot hold at float64's precision (rows 2^200 apart), far from
    1 (2^-900, 2^400), all zero, or zero but for one cell."""
    shape = (256, 128)
    u0, f = random_field(shape, 621, -1, 1), random_field(shape, 622, -1, 1)
    rows = 2.0 ** (-200.0 * np.arange(shape[0]) / shape[0])[:, None]
    if kind == "zero":
        u0, f = 0 * u0, 0 * f
    elif kind == "rows":
        u0, f = u0 * rows, f * rows
    elif kind == "tiny":
        u0, f = u0 * 2.0 ** -900, f * 2.0 ** -900
    elif kind == "huge":
        u0, f = u0 * 2.0 ** 400, f * 2.0 ** 400
    else:
        u0, f = 0 * u0, 0 * f
        f[100, 77] = 3.0
    a, b = (_cycles(cuda_lib, shape, path, u0, f) for path in (0, 1))
    assert np.all(np.isfinite(a))
    assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
    if kind == "zero":
        assert not a.any()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_tile_float64_nonfinite(cuda_lib, bad):
    fas = cuda_lib
    shape = (128, 128)
    f = random_field(shape, 631)
    f[70, 3] = bad
    ctx = fas.fas_create(fas.make_params(shape, 1.0 / 128, beta=1e-3))
    with pytest.raises(fas.FasError) as e:
        fas.fas_solve(ctx, _t(np.zeros(shape)), _t(f))
    assert e.value.status == fas.FAS_ENONFINITE


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,bc,nu,contrast", [
    ((128, 128), (N_,) * 4, 2, 1.0), ((32, 64), (D_, N_, N_, D_), 2, 1.0), ((16, 16), (N_,) * 4, 1, 1.0),
    ((256, 64), (D_,) * 4, 3, 1e4), ((64, 512), (N_, D_, D_, N_), 2, 1e4), ((256, 512), (N_,) * 4, 4, 1e2)])
def test_tile_kernels_per_cell_diffusivity(cuda_lib, shape, bc, nu, contrast, precision):
    """The same with a per-cell diffusivity (weights as 62-bit fractions in float64), up to a jump of 1e4."""
    fas = cuda_lib
    u0, f = random_field(shape, 651, -1, 1), noisy_cos_mode(shape, 652)
    kappa = _t(0.5 + random_field(shape, 653) * np.where(np.arange(shape[1]) < shape[1] // 3, contrast, 1.0)[None, :])
    out = []
    for path in (0, 1):
        ctx = fas.fas_create(fas.make_params(shape, 1.0 / max(shape), beta=2e-3, path=path, bc=bc, nu1=nu, nu2=nu,
                                             precision=precision), kappa=kappa)
        u, ft = _t(u0), _t(f)
        for _ in range(3):
            fas.fas_vcycle(ctx, u, ft)
        out.append(u.cpu().numpy())
    if precision == 1:
        np.testing.assert_array_equal(out[0], out[1])
    else:
        assert np.max(np.abs(out[0] - out[1])) <= 1e-12 * np.max(np.abs(out[1]))


@pytest.mark.parametrize("shape,nu", [((128, 128), 2), ((256, 256), 2), ((512, 1024), 3)])
def test_tile_kernels_repeat(cuda_lib, shape, nu):
    """A warp that is late in the tau correction must not see the first phase of the others: twenty runs of three
    float32 cycles, bit for bit."""
    u0, f = random_field(shape, 661, -1, 1), noisy_cos_mode(shape, 662)
    kw = dict(nu1=nu, nu2=nu, precision=1, inner_cycles=2)
    b = _cycles(cuda_lib, shape, 1, u0, f, **kw)
    for _ in range(20):
        np.testing.assert_array_equal(_cycles(cuda_lib, shape, 0, u0, f, **kw), b)
