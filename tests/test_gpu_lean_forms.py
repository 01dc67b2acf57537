"""Every launch form of the lean mixed column gives the same bits, at the level counts and grid
sizes where its runs of levels, pairs of levels and partial warps end."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topo_m", [0.0, 1500.0])
@pytest.mark.parametrize("bisections,nlev", [(0, 2), (0, 9), (1, 33), (0, 90), (1, 256)])
def test_forms_agree(gpu, bisections, nlev, topo_m):
    """R2B0 has 80 cells (two and a half warps of columns); 2 levels leave most warps of a tile
    without a run, 256 are the most a grid can have."""
    C = gpu
    dt = 100.0
    grid = C.icon_grid_build(2, bisections, nlev)
    want = None
    for form in C.LEAN_SHAPES:
        st = C.icon_state_init_ex(grid, 5, C.ICON_CASE_JET, noise_K=0.1, precision=C.ICON_MIXED, topo_height_m=topo_m,
                                  topo_radius_m=1.5e6 if topo_m else 0.0)
        C.icon_state_set_tiling(st, C.KIND_MX_LEAN, *form)
        for _ in range(2):
            C.icon_dycore_step(st, dt, 5)
        got = {f: C.icon_state_copy_field(st, grid, nlev, f) for f in C.FIELDS}
        C.icon_state_free(st)
        assert all(np.all(np.isfinite(x)) for x in got.values())
        if want is None:
            want = got
        for f in got:
            assert np.array_equal(got[f], want[f]), (form, f)
    C.icon_grid_free(grid)
