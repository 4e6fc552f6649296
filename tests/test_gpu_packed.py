"""The collisions on pairs of sites (packed FP32 instructions) against the ones on
single sites: every variant of the step from one random state far from
equilibrium, four steps, bit for bit.  Single-site forms remain in the tiled
small-list variant, in FP32 register-staged steps of periodic channels and in the
one-site-wide FP32 step of open channels; the others are packed."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


@pytest.fixture(scope="module")
def L():
    from paper_2005_09323_gb300 import build, lbmrare
    build.build()
    lbmrare.lib()
    return lbmrare


@pytest.mark.parametrize("is_open", [False, True], ids=["periodic", "open"])
@pytest.mark.parametrize("collision", ["bgk", "cm"])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_every_variant_agrees_on_random_states(L, storage, collision, is_open):
    nx, ny, n = 264, 40, 2
    kw = dict(obstacle=(100, 14, 9, 11), tau=0.62, storage=storage, max_steps=8, collision=collision, omega_bulk=1.1,
              omega_3=0.9, omega_4=1.2)
    if is_open:
        kw.update(open_x=1, u_in=0.05, grid=(16, 8, 6, 6), sponge_len=60, sponge_tau=0.95)
    else:
        kw.update(gx=3e-5, gy=-2e-5)
    rng = np.random.default_rng(17)
    start = [W * (1 + 0.6 * rng.uniform(-1, 1, (9, ny, nx))) for _ in range(n)]
    got = {}
    for v in range(L.lbm_step_variant_count()):
        if L.lbm_step_variant_info(v)[0] != L.STORAGE[storage]:
            continue
        e = L.lbm_ensemble_create(L.config(nx, ny, **kw), n, 1, torch.cuda.current_stream())
        try:
            try:
                L.lbm_ensemble_set_variant(e, v)
            except L.LbmError:
                continue
            for c in range(n):
                L.lbm_ensemble_set_populations(e, c, start[c])
            L.lbm_ensemble_step(e, 4)
            got[L.lbm_step_variant_kind(v), L.lbm_step_variant_info(v)[1:]] = [
                L.lbm_ensemble_get_populations(e, c, nx, ny) for c in range(n)]
        finally:
            L.lbm_ensemble_destroy(e)
    assert len(got) >= 3 and any(k == 3 for k, _ in got)
    ref = next(iter(got.values()))
    assert np.all(np.isfinite(ref[0])) and np.abs(ref[0] - start[0]).max() > 1e-3
    for key, pops in got.items():
        assert all(np.array_equal(a, b) for a, b in zip(pops, ref)), key
