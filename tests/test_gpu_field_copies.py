"""Copies between a state's device layouts and host order return what was set, to the bit: to
pageable and to pinned buffers, at entity counts that end inside a tile of 32, at the smallest and
the largest number of levels, and with no device memory left for a packed buffer."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(0, 2), (0, 31), (0, 33), (1, 256)]


def _pinned(shape):
    import torch
    return torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()


def _values(rng, shape):
    return rng.uniform(0.5, 1.5, shape).astype(np.float32).astype(np.float64)   # exact in either precision


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bis,nlev", SIZES)
def test_fields_return_as_set(gpu, bis, nlev, precision):
    C = gpu
    rng = np.random.default_rng(5)
    grid = C.icon_grid_build(2, bis, nlev)
    st = C.icon_state_init_ex(grid, 1, C.ICON_CASE_JET, precision=C.ICON_MIXED if precision == "mixed" else C.ICON_FP64)
    try:
        for f in ("vn", "w", "rho", "theta_v", "exner"):
            shape = C.icon_state_copy_field(st, grid, nlev, f).shape
            for src_pinned in (False, True):
                x = _values(rng, shape)
                if src_pinned:
                    buf = _pinned(shape)
                    buf[...] = x
                else:
                    buf = x
                C.icon_state_set_field(st, grid, nlev, f, buf)
                assert np.array_equal(C.icon_state_copy_field(st, grid, nlev, f), x), f
                assert np.array_equal(C.icon_state_copy_field(st, grid, nlev, f, _pinned(shape)), x), f
    finally:
        C.icon_state_free(st)
        C.icon_grid_free(grid)


@pytest.mark.parametrize("refuse", [False, True])
@pytest.mark.parametrize("bis,nlev", SIZES)
def test_tracers_return_as_set(gpu, bis, nlev, refuse):
    """`refuse`: the allocator has nothing left once the state is made."""
    import torch
    import paper_2511_02021_gb300 as P
    C = gpu
    rng = np.random.default_rng(6)
    full = [False]

    def alloc(n):
        return 0 if full[0] else torch.cuda.caching_allocator_alloc(n, 0, torch.cuda.current_stream())

    C.icon_set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        grid = C.icon_grid_build(2, bis, nlev)
        st = C.icon_state_init_ex(grid, 1, C.ICON_CASE_JET)
        C.icon_state_add_tracers(st, 2)
        full[0] = refuse
        nc = C.icon_grid_counts(grid)[0]
        want = []
        for t in range(2):
            x = rng.uniform(0.0, 1.0, (nc, nlev))
            buf = x
            if t:
                buf = _pinned(x.shape)
                buf[...] = x
            C.icon_state_set_tracer(st, grid, nlev, t, buf)
            want.append(x)
        for t in range(2):
            assert np.array_equal(C.icon_state_copy_tracer(st, grid, nlev, t), want[t]), t
        C.icon_state_free(st)
        C.icon_grid_free(grid)
    finally:
        P.use_torch_allocator(0)


def test_domain_field_without_room_for_the_global_order(gpu):
    import torch
    import paper_2511_02021_gb300 as P
    C = gpu
    N, full = 33, [0]

    def alloc(n):
        if full[0] and n >= full[0]:
            return 0
        return torch.cuda.caching_allocator_alloc(n, 0, torch.cuda.current_stream())

    C.icon_set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        grid = C.icon_grid_build(2, 2, N)
        src = C.icon_state_init_ex(grid, 5, C.ICON_CASE_JET, noise_K=0.1)
        dom = C.icon_domain_create(src, 4, 3)
        C.icon_domain_step(dom, 300.0, 5)
        want = {f: C.icon_domain_copy_field(dom, grid, N, f) for f in C.FIELDS}
        for f, x in want.items():
            full[0] = x.nbytes                    # the global order does not fit, a part's field does
            assert np.array_equal(C.icon_domain_copy_field(dom, grid, N, f), x), f
        full[0] = 0
        C.icon_domain_free(dom)
        C.icon_state_free(src)
        C.icon_grid_free(grid)
    finally:
        P.use_torch_allocator(0)
