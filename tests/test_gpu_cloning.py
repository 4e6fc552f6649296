"""The cloning step's reductions and copies at the sizes where their kernels
change form: moments of states whose sums leave one thread's few values, or
FP32's range; more than 64 changing slots and every width of the snapshot bank."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
W32 = W.astype(np.float32).astype(np.float64)
CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])


@pytest.fixture(scope="module")
def L():
    from paper_2005_09323_gb300 import build, lbmrare
    build.build()
    lbmrare.lib()
    return lbmrare


def stored(f, storage):
    """the stored populations less their rest weights, exactly"""
    if storage == "fp32":
        return (f.astype(np.float32) - W.astype(np.float32)[:, None, None]).astype(np.float64)
    dt = torch.float16 if storage == "fp16" else torch.bfloat16
    return torch.from_numpy((f - W[:, None, None]).astype(np.float32)).to(dt).double().numpy()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(2048, 512), (200, 37)])
def test_moments_of_mixed_magnitudes_are_the_exact_sums(L, storage, nx, ny):
    """Random deviations from 1e-9 to 0.3 of both signs (momentum near zero against
    the sum of the magnitudes).  A stored deviation is a multiple of 2^-30 (FP32) or
    has at most 11 significant bits, so FP64 holds the sums of these sizes to the last
    bit or two: 8 ulp of the sum of magnitudes over 2^20 for the momenta (an FP32 sum
    would be off by 2^-24 of it), 4 ulp of the mass"""
    rng = np.random.default_rng(nx)
    dev = np.exp(rng.uniform(np.log(1e-9), np.log(0.3), (9, ny, nx))) * rng.choice([-1.0, 1.0], (9, ny, nx))
    f = W[:, None, None] + dev
    e = L.lbm_ensemble_create(L.config(nx, ny, tau=0.6, max_steps=1, storage=storage), 1, 1,
                              torch.cuda.current_stream())
    try:
        L.lbm_ensemble_set_populations(e, 0, f)
        m, px, py = L.lbm_ensemble_moments(e, 1)
    finally:
        L.lbm_ensemble_destroy(e)
    g = stored(f, storage)
    per_q = [math.fsum(x.ravel()) for x in g]
    total = np.abs(g).sum()
    assert abs(px[0] - math.fsum(CX * per_q)) <= 8 * np.spacing(total) / 2 ** 20
    assert abs(py[0] - math.fsum(CY * per_q)) <= 8 * np.spacing(total) / 2 ** 20
    ref = math.fsum(per_q) + nx * ny * math.fsum(W32)
    assert abs(m[0] - ref) <= 4 * np.spacing(ref)


def test_moments_beyond_the_range_of_fp32_sums(L):
    """populations whose FP32 sum is infinite: summed in FP64"""
    nx, ny = 64, 16
    f = np.broadcast_to(W[:, None, None], (9, ny, nx)).copy()
    f[0, :, ::2] = 2e38
    f[1, 3:9, :] = 3e38
    e = L.lbm_ensemble_create(L.config(nx, ny, tau=0.6, max_steps=1), 1, 1, torch.cuda.current_stream())
    try:
        L.lbm_ensemble_set_populations(e, 0, f)
        m, px, py = L.lbm_ensemble_moments(e, 1)
    finally:
        L.lbm_ensemble_destroy(e)
    f32 = f.astype(np.float32).astype(np.float64)
    assert abs(m[0] / f32.sum() - 1) < 1e-12
    assert abs(px[0] / (CX[:, None, None] * f32).sum() - 1) < 1e-12
    assert py[0] == pytest.approx((CY[:, None, None] * f32).sum(), abs=1e-6)


@pytest.mark.parametrize("n_snap", [1, 10, 11, 16])
def test_many_clones_and_snapshots_match_oracle(L, orc, n_snap):
    """67 of 70 slots become perturbed copies of three parents"""
    n, nx, ny, obstacle = 70, 72, 18, (20, 6, 5, 5)
    kw = dict(obstacle=obstacle, tau=0.6, gx=2e-5, gy=-5e-6)
    oc = orc.cfg(nx, ny, **kw)
    e = L.lbm_ensemble_create(L.config(nx, ny, max_steps=20, n_snapshots=n_snap, init_amp=0.01, **kw), n, 2,
                              torch.cuda.current_stream())
    try:
        L.lbm_ensemble_step(e, 10)
        at10 = {c: orc.run(oc, orc.init(oc, 2, c, 0.01), 10)[0] for c in range(max(n_snap, 3))}
        L.lbm_ensemble_set_snapshots(e, list(range(n_snap)))
        parent = np.arange(n) % 3
        L.lbm_ensemble_clone(e, torch.tensor(parent, dtype=torch.int32, device="cuda"), 0.002, 77, 5)
        snaps = np.stack([at10[c] for c in range(n_snap)])
        for s in (3, 31, 32, 62, 63, 64, 66, 67, 69):
            ref = orc.perturb(oc, at10[s % 3], snaps, orc.perturb_alphas(77, 5, s, n_snap), 0.002)
            got = L.lbm_ensemble_get_populations(e, s, nx, ny)
            assert np.abs(got - ref).max() / np.abs(ref).max() < 1e-6, s
        for s in range(3):
            got = L.lbm_ensemble_get_populations(e, s, nx, ny)
            assert np.abs(got - at10[s]).max() / np.abs(at10[s]).max() < 1e-6
    finally:
        L.lbm_ensemble_destroy(e)


def test_observables_of_a_square_beyond_shared_memory(L, orc):
    """6200 nodes: not staged.  Bounds as for the small squares: pressures 1e-6
    relative, shears 1e-3 of the largest"""
    nx, ny, obstacle, steps = 2048, 108, (200, 4, 1500, 100), 5
    oc = orc.cfg(nx, ny, obstacle=obstacle, tau=0.6, gx=2e-5)
    e = L.lbm_ensemble_create(L.config(nx, ny, obstacle=obstacle, tau=0.6, gx=2e-5, max_steps=steps, init_amp=0.02), 1,
                              4, torch.cuda.current_stream())
    try:
        L.lbm_ensemble_set_observables(e, True)
        L.lbm_ensemble_step(e, steps)
        got = np.zeros((1, steps, 4))
        L.lbm_ensemble_observables(e, 0, steps, got)
    finally:
        L.lbm_ensemble_destroy(e)
    f = orc.init(oc, 4, 0, 0.02)
    for t in range(steps):
        f, _, _ = orc.step(oc, f)
        ref = np.array(orc.observables(oc, f))
        assert np.abs(got[0, t, :2] - ref[:2]).max() < 1e-6 * np.abs(ref[:2]).max()
        assert np.abs(got[0, t, 2:] - ref[2:]).max() < 1e-3 * np.abs(ref[2:]).max()
