"""A forced tile selects the kernel that runs: on small grids, where the vertices and the edge diagnostics
share a launch while their tiles are automatic, and on grids above that, where every kind has
its own. The results are the same bits whichever runs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FIELDS = ("vn", "w", "rho", "theta_v", "exner", "mflx", "wflx")


def _run(C, grid, nlev, topo_m, tiles, dt):
    """(fields after two steps, launches per kind of a third) with {kind: tile} forced"""
    st = C.icon_state_init_ex(grid, 9, C.ICON_CASE_JET, noise_K=0.1, precision=C.ICON_MIXED, topo_height_m=topo_m,
                              topo_radius_m=1.5e6 if topo_m else 0.0)
    try:
        for kind, tile in tiles.items():
            C.icon_state_set_tiling(st, kind, *tile)
        for _ in range(2):
            C.icon_dycore_step(st, dt, 5)
        for kind, tile in tiles.items():
            assert C.icon_state_tiling(st, kind) == tile
        out = {f: C.icon_state_copy_field(st, grid, nlev, f) for f in FIELDS}
        assert all(np.all(np.isfinite(x)) for x in out.values())
        return out, list(C.icon_dycore_step_profile(st, dt, 5)[1])
    finally:
        C.icon_state_free(st)


def _same(a, b):
    return all(np.array_equal(a[f], b[f]) for f in FIELDS)


@pytest.mark.parametrize("topo_m", [0.0, 1500.0])
@pytest.mark.parametrize("bisections,nlev", [(1, 9), (3, 33)])
def test_forced_tiles_keep_the_small_grids_launches_apart(gpu, bisections, nlev, topo_m):
    C = gpu
    grid = C.icon_grid_build(2, bisections, nlev)
    try:
        want, n = _run(C, grid, nlev, topo_m, {}, 100.0)
        assert n[C.KIND_MX_VERTEX] == 10 and n[C.KIND_MX_EDGE] == 0          # one launch per stage for both
        for tiles in ({C.KIND_MX_VERTEX: (32, 64)}, {C.KIND_MX_EDGE: (16, 512)},
                      {C.KIND_MX_VERTEX: (8, 256), C.KIND_MX_EDGE: (32, 128)},
                      {C.KIND_MX_VERTEX: (16, 128), C.KIND_MX_EDGE: (8, 64), C.KIND_MX_EDGE_TEND: (16, 512)}):
            got, n = _run(C, grid, nlev, topo_m, tiles, 100.0)
            assert n[C.KIND_MX_VERTEX] == 10 and n[C.KIND_MX_EDGE] == 10, tiles
            assert _same(got, want), tiles
    finally:
        C.icon_grid_free(grid)


@pytest.mark.parametrize("topo_m", [0.0, 1500.0])
def test_tiles_of_larger_grids_agree(gpu, topo_m):
    C = gpu
    nlev, kinds = 33, (C.KIND_MX_VERTEX, C.KIND_MX_EDGE, C.KIND_MX_CELL_KE, C.KIND_MX_EDGE_TEND, C.KIND_MX_DIFF_VERTEX)
    grid = C.icon_grid_build(2, 5, nlev)
    try:
        want, n = _run(C, grid, nlev, topo_m, {}, 40.0)
        assert n[C.KIND_MX_VERTEX] == 10 and n[C.KIND_MX_EDGE] == 10
        for tile in ((32, 128), (16, 512), (8, 64), (32, 512), (8, 256)):
            got, _ = _run(C, grid, nlev, topo_m, {k: tile for k in kinds}, 40.0)
            assert _same(got, want), tile
    finally:
        C.icon_grid_free(grid)
