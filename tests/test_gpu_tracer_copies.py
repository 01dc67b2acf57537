"""Tracers cross to and from host memory row by row where that is the faster way and as one packed
run elsewhere: the small ones take no device buffer, and both ways return what was set."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bisections,nlev,rows_in,rows_out", [
    (0, 20, True, True), (1, 90, True, True), (2, 20, False, True), (2, 128, True, True), (2, 8, True, True),
    (3, 4, True, True), (3, 47, False, False), (3, 128, False, True), (3, 90, False, False)])
def test_pageable_tracers(gpu, bisections, nlev, rows_in, rows_out):
    import torch
    import paper_2511_02021_gb300 as P
    C = gpu
    calls = [0]

    def alloc(n):
        calls[0] += 1
        return torch.cuda.caching_allocator_alloc(n, 0, torch.cuda.current_stream())

    C.icon_set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        grid = C.icon_grid_build(2, bisections, nlev)
        st = C.icon_state_init_ex(grid, 1, C.ICON_CASE_JET)
        C.icon_state_add_tracers(st, 2)
        x = np.random.default_rng(7).uniform(0.0, 1.0, (C.icon_grid_counts(grid)[0], nlev))
        calls[0] = 0
        C.icon_state_set_tracer(st, grid, nlev, 1, x)
        assert (calls[0] == 0) == rows_in
        calls[0] = 0
        assert np.array_equal(C.icon_state_copy_tracer(st, grid, nlev, 1), x)
        assert (calls[0] == 0) == rows_out
        assert not C.icon_state_copy_tracer(st, grid, nlev, 0).any()
        C.icon_state_free(st)
        C.icon_grid_free(grid)
    finally:
        P.use_torch_allocator(0)


@pytest.mark.parametrize("bisections,nlev", [(0, 9), (0, 16), (1, 33), (2, 8), (3, 48), (3, 47)])
def test_pinned_tracers(gpu, bisections, nlev):
    import torch
    C = gpu
    grid = C.icon_grid_build(2, bisections, nlev)
    st = C.icon_state_init_ex(grid, 1, C.ICON_CASE_JET)
    try:
        C.icon_state_add_tracers(st, 2)
        n = C.icon_grid_counts(grid)[0]
        x = torch.rand((n, nlev), dtype=torch.float64).pin_memory().numpy()
        y = torch.empty((n, nlev), dtype=torch.float64, pin_memory=True).numpy()
        C.icon_state_set_tracer(st, grid, nlev, 1, x)
        C._check(C._lib.icon_state_copy_tracer(st, 1, y.ctypes.data, y.size))
        assert np.array_equal(x, y)
        assert not C.icon_state_copy_tracer(st, grid, nlev, 0).any()
    finally:
        C.icon_state_free(st)
        C.icon_grid_free(grid)
