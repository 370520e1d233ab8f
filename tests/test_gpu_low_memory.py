"""Contexts created with too little free device memory for the second buffers of the fused kernels: they run the
per-operation kernels instead, give back what they had taken, and give the results of that path."""
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _used(fas, params):
    before = _free()
    ctx = fas.fas_create(params)
    used = before - _free()
    fas.fas_destroy(ctx)
    return used


class _Leave:
    """Takes the free device memory but for `nbytes`."""

    def __init__(self, nbytes):
        import torch
        torch.cuda.empty_cache()
        self.t = torch.empty((_free() - nbytes) // (2 * MB) * (2 * MB), dtype=torch.uint8, device="cuda")

    def release(self):
        import torch
        self.t = None
        torch.cuda.empty_cache()


@pytest.mark.parametrize("shape,precision,path0", [((512, 512, 512), 1, "column kernels"), ((4096, 4096), 0, "tiles")])
def test_fallback_without_second_buffers(cuda_lib, shape, precision, path0):
    import torch
    fas = cuda_lib

    def params(path):
        return fas.make_params(shape, 1.0 / shape[-1], beta=1e-3, precision=precision, path=path)

    fas.fas_destroy(fas.fas_create(params(0)))  # the library's own memory
    need, basic = _used(fas, params(0)), _used(fas, params(1))
    assert need > basic + 64 * MB, path0
    hog = _Leave(need - 32 * MB)
    try:
        ctx = fas.fas_create(params(0))
        left = _free()
    finally:
        hog.release()
    # all but one field of the finest level (the sweep-fused 3D kernel's, in float32) has been given back; the smallest
    # buffers in question take 64 MB, and free memory moves by some 20 MB between the measurements
    cells = 1
    for n in shape:
        cells *= n
    assert left >= need - 32 * MB - basic - (4 * cells if len(shape) == 3 else 0) - 40 * MB
    gen = torch.Generator("cuda").manual_seed(761)
    u0 = torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen)
    f = torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen)
    out = []
    for c in (ctx, fas.fas_create(params(1))):
        u = u0.clone()
        for _ in range(2):
            fas.fas_vcycle(c, u, f)
        out.append(u)
        fas.fas_destroy(c)
    assert torch.equal(out[0], out[1])


def test_later_buffers_fit(cuda_lib):
    """A context whose second buffers would take the room that its heat right-hand side needs later."""
    import torch
    fas = cuda_lib
    shape, dt = (4096, 4096), 1e-4
    field = 8 * shape[0] * shape[1]

    def params(path):
        return fas.make_params(shape, 1.0 / shape[-1], alpha=1.0, beta=dt, path=path)

    fas.fas_destroy(fas.fas_create(params(0)))
    need, basic = _used(fas, params(0)), _used(fas, params(1))
    leave = need + field // 2
    assert leave > basic + field + 32 * MB
    gen = torch.Generator("cuda").manual_seed(762)
    u0 = torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen)
    u, ref = u0.clone(), u0.clone()
    hog = _Leave(leave)
    try:
        ctx = fas.fas_create(params(0))
        fas.fas_heat_run(ctx, u, None, dt, 1)
    finally:
        hog.release()
    fas.fas_destroy(ctx)
    ctx = fas.fas_create(params(1))
    fas.fas_heat_run(ctx, ref, None, dt, 1)
    fas.fas_destroy(ctx)
    assert torch.equal(u, ref)
