"""The row-streaming step (two steps per pass over memory) against the
register-staged step with the same drag segments: the same arithmetic in the
same order, so populations and drag agree bit for bit (no tolerance).  Sizes at
the edges: one warp and sixteen, a last warp of few sites, two-row channels'
neighbours, obstacles at the seam, on a wall, one cell large and over most of a
row, and step counts with every remainder modulo four."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [  # clones, nx, ny, obstacle, step counts
    (3, 200, 37, (60, 11, 9, 14), (4, 5, 6, 7)),
    (5, 8, 5, (0, 0, 0, 0), (8,)),
    (2, 16, 4, (4, 0, 4, 2), (12,)),
    (4, 2048, 65, (500, 28, 64, 36), (13,)),
    (40, 512, 17, (126, 5, 4, 4), (9,)),
    (2, 64, 20, (1, 3, 20, 4), (8,)),
    (2, 72, 20, (60, 5, 11, 3), (12,)),
    (3, 136, 9, (1, 1, 1, 1), (16,)),
]


@pytest.fixture(scope="module")
def L():
    from paper_2005_09323_gb300 import build, lbmrare
    build.build()
    lbmrare.lib()
    return lbmrare


def variant(L, storage, kind):
    """the streaming variant, or the register-staged one of its vector width with four warps"""
    st = L.STORAGE[storage]
    vec = 4 if storage == "fp32" else 8
    for v in range(L.lbm_step_variant_count()):
        s, ve, warps = L.lbm_step_variant_info(v)
        if s == st and L.lbm_step_variant_kind(v) == kind and ve == vec and (kind != 0 or warps == 4):
            return v
    raise AssertionError("variant not compiled")


def run(L, cfg, n, steps, v=None):
    e = L.lbm_ensemble_create(cfg, n, 5, torch.cuda.current_stream())
    try:
        if v is not None:
            L.lbm_ensemble_set_variant(e, v)
        l0 = L.lbm_launch_count()
        for s in steps:
            L.lbm_ensemble_step(e, s)
        launches = L.lbm_launch_count() - l0
        drag = np.zeros((n, sum(steps)))
        L.lbm_ensemble_drag(e, 0, sum(steps), drag)
        pops = [L.lbm_ensemble_get_populations(e, c, cfg.nx, cfg.ny) for c in sorted({0, n // 2, n - 1})]
        return drag, pops, launches
    finally:
        L.lbm_ensemble_destroy(e)


@pytest.mark.parametrize("storage,shift", [("fp32", 0), ("fp16", 3), ("bf16", 0)])
@pytest.mark.parametrize("collision", ["bgk", "cm"])
def test_stream_is_the_single_step_bit_for_bit(L, storage, shift, collision):
    for n, nx, ny, ob, steps in SHAPES:
        cfg = L.config(nx, ny, obstacle=ob, tau=0.56, gx=2e-6, gy=-1e-6, storage=storage, shift_exp=shift, max_steps=64,
                       collision=collision, omega_bulk=1.1, omega_3=0.9, omega_4=1.2)
        a, b = (run(L, cfg, n, steps, variant(L, storage, k)) for k in (0, 3))
        assert np.array_equal(a[0], b[0]), (nx, ny)
        assert all(np.array_equal(x, y) for x, y in zip(a[1], b[1])), (nx, ny)


OPEN_SHAPES = [  # clones, nx, ny, obstacle, grid, sponge columns, step counts
    (3, 203, 37, (90, 11, 9, 14), (16, 8, 8, 8), 50, (4, 5, 6, 7)),
    (2, 64, 12, (0, 0, 0, 0), (0, 0, 0, 0), 16, (8,)),
    (7, 513, 33, (248, 9, 16, 9), (16, 8, 8, 8), 128, (9,)),
    (4, 517, 129, (248, 56, 16, 16), (2, 8, 8, 8), 128, (13, 4)),  # the grid at the inlet; padded last vector
    (5, 131, 17, (60, 5, 4, 4), (0, 0, 0, 0), 0, (9, 4)),
    (2, 1025, 60, (500, 20, 20, 20), (30, 10, 6, 6), 200, (12,)),
    (3, 512, 40, (200, 0, 30, 9), (5, 3, 4, 4), 100, (8,)),        # the square on a wall
]


@pytest.mark.parametrize("storage,shift", [("fp32", 0), ("fp16", 3), ("bf16", 0)])
@pytest.mark.parametrize("collision", ["bgk", "cm"])
def test_open_stream_is_the_single_step_bit_for_bit(L, storage, shift, collision):
    for n, nx, ny, ob, grid, sponge, steps in OPEN_SHAPES:
        cfg = L.config(nx, ny, obstacle=ob, tau=0.56, storage=storage, shift_exp=shift, max_steps=64, open_x=1,
                       u_in=0.05, grid=grid, sponge_len=sponge, sponge_tau=0.9, collision=collision, omega_bulk=1.1,
                       omega_3=0.9, omega_4=1.2)
        a, b = (run(L, cfg, n, steps, variant(L, storage, k)) for k in (0, 3))
        assert np.array_equal(a[0], b[0]), (nx, ny)
        assert all(np.array_equal(x, y) for x, y in zip(a[1], b[1])), (nx, ny)


def test_default_streams_large_calls_only(L):
    """48 clones of 512 x 128 (10 rows a block) stream: 8 steps in 4 launches, as
    the single steps bit for bit; 16 clones step singly; so does a call of three
    steps, and every call while observables are recorded"""
    kw = dict(nx=512, ny=128, obstacle=(120, 56, 16, 16), tau=0.505, gx=1e-6, max_steps=64)
    drag, pops, launches = run(L, L.config(**kw), 48, (8, 3))
    assert launches == 4 + 1 + 3 + 1
    ref = run(L, L.config(**kw), 48, (8, 3), variant(L, "fp32", 0))
    assert np.array_equal(drag, ref[0]) and all(np.array_equal(x, y) for x, y in zip(pops, ref[1]))
    assert run(L, L.config(**kw), 16, (8,))[2] == 8 + 1
    e = L.lbm_ensemble_create(L.config(**kw), 48, 5, torch.cuda.current_stream())
    try:
        L.lbm_ensemble_set_observables(e, True)
        l0 = L.lbm_launch_count()
        L.lbm_ensemble_step(e, 8)
        assert L.lbm_launch_count() - l0 == 8 + 8 + 1
    finally:
        L.lbm_ensemble_destroy(e)


@pytest.mark.parametrize("nx", [64, 128])
def test_one_warp_rows_over_more_rows_than_blocks(L, nx):
    """rows of one warp, 15 (FP32) or 16 blocks an SM: spans of one, two and several
    rows, over clone boundaries"""
    for storage, n in (("fp32", 150), ("fp32", 290), ("fp16", 700)):
        cfg = L.config(nx, 16, obstacle=(20, 6, 5, 5), tau=0.56, gx=2e-6, storage=storage, max_steps=16)
        a, b = (run(L, cfg, n, (8,), variant(L, storage, k)) for k in (0, 3))
        assert np.array_equal(a[0], b[0]) and all(np.array_equal(x, y) for x, y in zip(a[1], b[1])), (storage, n)


OPEN_KW = dict(open_x=1, u_in=0.05, sponge_tau=1.0, collision="cm", tau=0.53)


@pytest.mark.parametrize("n,nx,ny,storage,kw,streams", [
    # measured slower streamed: large squares, few 16-bit rows, wide rows with few rows a
    # block, wide grids
    (15, 1024, 256, "fp32", dict(obstacle=(158, 28, 200, 200)), False),
    (48, 1024, 256, "fp32", dict(obstacle=(158, 28, 200, 200), collision="cm"), False),
    (190, 512, 128, "fp16", dict(obstacle=(98, 32, 64, 64)), False),
    (247, 256, 64, "bf16", dict(obstacle=(50, 16, 32, 32)), False),
    (4, 2049, 513, "fp32", dict(OPEN_KW, obstacle=(992, 224, 64, 64), grid=(64, 32, 32, 32), sponge_len=512), False),
    (4, 2049, 513, "fp16", dict(OPEN_KW, obstacle=(992, 224, 64, 64), grid=(64, 32, 32, 32), sponge_len=512), False),
    (127, 513, 129, "fp32", dict(OPEN_KW, collision="bgk", obstacle=(248, 56, 16, 16), grid=(16, 64, 8, 8),
                                 sponge_len=128), False),
    # measured faster streamed
    (64, 1024, 256, "fp32", dict(obstacle=(240, 112, 32, 32)), True),
    (16, 2048, 512, "fp16", dict(obstacle=(480, 224, 64, 64)), True),
    (64, 513, 129, "fp32", dict(OPEN_KW, obstacle=(248, 56, 16, 16), grid=(16, 8, 8, 8), sponge_len=128), True),
    (64, 513, 129, "bf16", dict(OPEN_KW, obstacle=(248, 56, 16, 16), grid=(16, 8, 8, 8), sponge_len=128), True),
    (494, 128, 64, "fp32", dict(obstacle=(32, 29, 6, 6), collision="cm"), True),
])
def test_default_streams_where_it_pays(L, n, nx, ny, storage, kw, streams):
    """eight steps: four launches streamed, eight single ones otherwise, and the drag's
    (the open channel's single steps also launch its outlet)"""
    cfg = L.config(nx, ny, max_steps=16, storage=storage, **dict(dict(tau=0.53), **kw))
    drag, pops, launches = run(L, cfg, n, (8,))
    assert launches == (5 if streams else 9 + (1 if kw.get("open_x") else 0))
    ref = run(L, cfg, n, (8,), variant(L, storage, 0))
    assert np.array_equal(drag, ref[0]) and all(np.array_equal(x, y) for x, y in zip(pops, ref[1]))


@pytest.mark.parametrize("n,nx,ny,storage,kw", [
    (28, 512, 128, "fp32", dict(obstacle=(122, 56, 16, 16))),  # six rows a block
    (152, 256, 64, "fp32", dict(obstacle=(50, 16, 32, 32))),   # streams faster, but not by default
    (52, 512, 128, "fp16", dict(obstacle=(122, 56, 16, 16))),
    (48, 512, 128, "fp32", dict(obstacle=(120, 56, 16, 16))),
    (30, 1024, 256, "fp32", dict(obstacle=(158, 28, 200, 200))),
])
def test_tuned_variant_is_the_one_that_runs(L, n, nx, ny, storage, kw):
    """eight steps take the launches of the variant that autotune returned; with three
    steps, and while observables are recorded, a streaming choice makes way for single
    steps, and the states do not depend on any of it"""
    cfg = L.config(nx, ny, max_steps=32, storage=storage, tau=0.53, **kw)
    ref = run(L, cfg, n, (8, 3, 4), variant(L, storage, 0))
    e = L.lbm_ensemble_create(cfg, n, 5, torch.cuda.current_stream())
    try:
        kind = L.lbm_step_variant_kind(L.lbm_ensemble_autotune(e))
        launches = []
        for steps, observe in ((8, False), (3, False), (4, True)):
            if observe:
                L.lbm_ensemble_set_observables(e, True)
            l0 = L.lbm_launch_count()
            L.lbm_ensemble_step(e, steps)
            launches.append(L.lbm_launch_count() - l0)
        assert launches[0] == {0: 9, 1: 9, 2: 5, 3: 5}[kind], kind
        assert launches[1] in (4, 2) and launches[2] == 4 + 4 + 1
        for c, f in zip(sorted({0, n // 2, n - 1}), ref[1]):
            assert np.array_equal(L.lbm_ensemble_get_populations(e, c, nx, ny), f)
    finally:
        L.lbm_ensemble_destroy(e)
