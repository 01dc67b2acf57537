"""Level-major fields in host order, on both sides of the line between blocks that take 32 levels and
blocks that take all of them (152 blocks of 32 cells: R2B2 has 40, R2B3 160), at levels that end
inside a chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bisections,nlev", [(0, 32), (1, 65), (2, 95), (2, 256), (3, 20), (3, 95), (3, 256)])
def test_level_major_fields_return_as_set(gpu, bisections, nlev):
    import torch
    C = gpu
    rng = np.random.default_rng(8)
    grid = C.icon_grid_build(2, bisections, nlev)
    st = C.icon_state_init_ex(grid, 1, C.ICON_CASE_JET, precision=C.ICON_MIXED)
    try:
        for f in ("w", "rho", "exner"):
            shape = C.icon_state_copy_field(st, grid, nlev, f).shape
            x = rng.uniform(0.5, 1.5, shape)
            C.icon_state_set_field(st, grid, nlev, f, x)
            assert np.array_equal(C.icon_state_copy_field(st, grid, nlev, f), x), f
            out = torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()
            assert np.array_equal(C.icon_state_copy_field(st, grid, nlev, f, out), x), f
    finally:
        C.icon_state_free(st)
        C.icon_grid_free(grid)
