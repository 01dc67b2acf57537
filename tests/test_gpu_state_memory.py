"""Device memory of an FP64 state: the fields it needs, counted, and no more, so that the largest
state a device holds does not shrink unnoticed."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topo_m", [0.0, 1500.0])
@pytest.mark.parametrize("bisections,nlev", [(2, 20), (3, 90)])
def test_fp64_state_holds_its_fields_and_no_more(gpu, bisections, nlev, topo_m):
    """9 edge, 23 cell and 4 vertex fields of ld levels (prognostics of S^n and S*, fluxes, the
    column's rows and operands, the stencils' outputs), 9 cell and 3 edge fields of metric terms
    over terrain; besides them tables of a value or a few per entity and per level."""
    import torch
    import paper_2511_02021_gb300 as P
    C = gpu
    total = [0]

    def alloc(n):
        total[0] += n
        return torch.cuda.caching_allocator_alloc(n, 0, torch.cuda.current_stream())

    C.icon_set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        grid = C.icon_grid_build(2, bisections, nlev)
        nc, ne, nv = C.icon_grid_counts(grid)
        total[0] = 0
        st = C.icon_state_init_ex(grid, 1, C.ICON_CASE_JET, topo_height_m=topo_m,
                                  topo_radius_m=1.5e6 if topo_m else 0.0)
        used = total[0]
        C.icon_state_free(st)
        C.icon_grid_free(grid)
    finally:
        P.use_torch_allocator(0)
    ld = (nlev + 1 + 31) // 32 * 32
    fields = ld * (9 * ne + 23 * nc + 4 * nv)
    tables = 6 * nc
    if topo_m:
        fields += ld * (9 * nc + 3 * ne)
        tables += nc + 2 * ne
    assert used <= 8 * (fields + tables) + (64 << 10)      # per-level tables and 256-byte blocks
