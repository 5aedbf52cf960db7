"""The kernel variants that sizes select (thin tiles, clustered snapshot, chunked column solver) at the
edges of their ranges, and the graphs that a handle and a batch keep, against the general path and the
FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1807_02137_gb300 import synth
from tests.gpu_common import gpu_solver, need_gpu, oracle_params, relmax, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def segmg():
    return need_gpu()


def image(n, m, seed):
    r = max(4, min(n, m) / 3)
    return synth.ellipses(n, m, 6, (r / 2, r), 5, 0.05, seed)[:2]


def levels_for(n, m):
    """Grids down to a coarsest one of at most 2048 cells, at least two."""
    l = 2
    while (n >> (l - 1)) * (m >> (l - 1)) > 2048:
        l += 1
    return l


# thin 8x32 / 32x8 tiles run where 4 blocks per SM hold them all (384x400 is below that line on 152
# SMs, 400x401 above it); sizes one beside a tile edge, and single rows and columns of tiles
@pytest.mark.parametrize("shape", [(7, 33), (9, 31), (33, 65), (31, 500), (500, 8), (129, 255), (384, 400), (400, 401)])
@pytest.mark.parametrize("precision", ["f32", "mixed", "f64"])
def test_thin_sweep_tiles_equal_per_phase_kernels(segmg, shape, precision):
    prec = {"f32": segmg.MG_F32, "mixed": segmg.MG_MIXED, "f64": segmg.MG_F64}[precision]
    img, mk = image(*shape, 3)
    outs = []
    for sm in (0, 1):
        s, _ = gpu_solver(segmg, img, mk, precision=prec, levels=levels_for(*shape), smoother=sm)
        s.set_bottom_kernel(False)
        s.begin_step()
        for _ in range(2):
            s.vcycle()
        outs.append(s.phi().cpu().numpy())
        s.close()
    assert np.isfinite(outs[0]).all() and np.array_equal(outs[0], outs[1])


# FP64: the snapshot on clusters of 8 or 4 blocks, the thin residual and the 8-, 4- and 2-wide sweep
# tiles against the oracle (tolerances of the existing V-cycle test)
@pytest.mark.parametrize("shape", [(9, 33), (33, 31), (64, 129), (130, 160), (257, 300)])
def test_fp64_thin_kernels_match_oracle(segmg, shape):
    img, mk = image(*shape, 4)
    s, p = gpu_solver(segmg, img, mk, precision=segmg.MG_F64, levels=levels_for(*shape))
    o = O.Solver(np.asarray(img, dtype=np.float64), mk, oracle_params(*shape, p))
    s.begin_step(); o.begin_step()
    for _ in range(2):
        rg, ro = s.vcycle(), o.vcycle()
        assert abs(rg - ro) <= 1e-8 * ro
    assert relmax(s.phi().cpu().numpy(), o.phi) < 1e-10
    s.close(); o.close()


# GSLINE-I: fewer rows than a chunk, a chunk's edge and one past it; the last block's idle lanes
@pytest.mark.parametrize("shape", [(5, 4), (16, 63), (17, 65), (33, 130), (65, 31)])
def test_gsline_chunk_edges_match_oracle(segmg, shape):
    img, mk = image(*shape, 5)
    s, p = gpu_solver(segmg, img, mk, precision=segmg.MG_F64, levels=levels_for(*shape), smoother=3)
    o = O.Solver(np.asarray(img, dtype=np.float64), mk, oracle_params(*shape, p))
    s.begin_step(); o.begin_step()
    for _ in range(2):
        rg, ro = s.vcycle(), o.vcycle()
        assert abs(rg - ro) <= 1e-8 * max(ro, 1e-6)
    assert relmax(s.phi().cpu().numpy(), o.phi) < 1e-10
    s.close(); o.close()


def test_kept_graphs_of_many_tau_values_give_a_fresh_handles_results(segmg):
    # seven steps that each reject one attempt take the handle through eight values of tau (more than
    # it keeps graphs of); images after that, with and without a rejected attempt, as fresh handles
    img, mk = image(150, 170, 6)
    img2, mk2 = image(150, 170, 7)
    s, p = gpu_solver(segmg, img, mk)
    for k in range(7):
        s.inject_divergence(2)
        s.solve_step(1e-6, 40)
        assert s.stats()["tau"] <= p.tau * 0.5 ** (k + 1)
    for inject in (0, 2, 0):
        t = torch.as_tensor(np.ascontiguousarray(img2), dtype=torch.float32, device="cuda")
        s.reset(t, mk2)
        f, _ = gpu_solver(segmg, img2, mk2)
        for h in (s, f):
            if inject:
                h.inject_divergence(inject)
            h.solve_step(1e-6, 40)
            h.solve_step(1e-6, 40)
        assert s.stats()["tau"] == f.stats()["tau"]
        assert np.array_equal(s.phi().cpu().numpy(), f.phi().cpu().numpy())
        f.close()
    s.close()


def test_batch_restart_rounds_equal_individual_solves(segmg):
    # a cap on the V-cycles of an attempt that some images keep and others do not: these restart, as
    # a graph of their own, and the next image set starts from tau again
    shapes = [(64, 64), (96, 80), (128, 128), (40, 200), (160, 160)]
    pairs = [image(n, m, 40 + q) for q, (n, m) in enumerate(shapes)]
    imgs = [torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a, _ in pairs]
    mks = [mk for _, mk in pairs]
    free = []
    for a, mk in pairs:
        s, _ = gpu_solver(segmg, a, mk)
        free.append(s.solve_step(1e-6, 60)[0])
        s.close()
    cap = sorted(free)[2]
    b = segmg.Batch(imgs, mks, [segmg.default_params(n, m) for n, m in shapes])
    for again in range(2):
        if again:
            b.reset(imgs, mks)
        cyc, rho = b.solve_step(1e-6, cap)
        for q, (a, mk) in enumerate(pairs):
            s, _ = gpu_solver(segmg, a, mk)
            c, r = s.solve_step(1e-6, cap)
            assert cyc[q] == c and rho[q] == r and b.solver(q).stats()["tau"] == s.stats()["tau"]
            assert np.array_equal(b.solver(q).phi().cpu().numpy(), s.phi().cpu().numpy())
            s.close()
    b.close()


# the tail kernel (one block for the smallest grids: FP64 storage, the Rada-Chen model) against the
# per-grid kernels, down to what can be read of every grid; its first grid one cell wide of a limit,
# long and thin, and as wide as it takes
@pytest.mark.parametrize("kw", [{"precision": 1}, {"precision": 1, "model": 1}, {"model": 1},
                                {"precision": 2, "model": 1}])
@pytest.mark.parametrize("shape,levels,nu", [((130, 97), 6, (2, 2)), ((64, 64), 4, (1, 3)), ((33, 67), 5, (3, 1)),
                                             ((20, 125), 4, (2, 1))])
def test_tail_kernel_equals_per_grid_kernels(segmg, kw, shape, levels, nu):
    names = {0: segmg.MG_F32, 1: segmg.MG_F64, 2: segmg.MG_MIXED}
    par = {"precision": names[kw.get("precision", 0)], "model": segmg.MG_MODEL_RC if kw.get("model") else segmg.MG_MODEL_SC}
    img, mk = image(*shape, 8)
    outs, count = [], []
    for on in (True, False):
        s, p = gpu_solver(segmg, img, mk, levels=levels, nu1=nu[0], nu2=nu[1], **par)
        s.set_bottom_kernel(on)
        s.begin_step()
        c0 = s.stats()["launches"]
        rho = [s.vcycle() for _ in range(3)]
        count.append(s.stats()["launches"] - c0)
        outs.append([rho] + [s.level(l, f).cpu().numpy() for l in range(levels) for f in ("phi", "rhs", "G")
                             if not (f == "G" and l == levels - 1) and not (f == "rhs" and l == 0)])
        s.close()
    assert count[0] < count[1]
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


# set-up and step start on 32 x 32 tiles: single rows and columns, one beside a tile edge, grids
# narrower than the blur's reach (sigma 1: 3, sigma 5: 15 cells), more markers than a chunk of 32
@pytest.mark.parametrize("shape,sigma,k", [((1, 40), 1.0, 3), ((33, 31), 1.0, 5), ((2, 65), 5.0, 4), ((70, 3), 5.0, 3),
                                           ((97, 130), 2.0, 70)])
@pytest.mark.parametrize("model", [0, 1])
def test_setup_tiles_match_oracle(segmg, shape, sigma, k, model):
    n, m = shape
    rng = np.random.default_rng(n + m)
    img = rng.random((n, m))
    mk = np.stack([rng.uniform(0, m - 1, k), rng.uniform(0, n - 1, k)], axis=1)
    s, p = gpu_solver(segmg, img, mk, precision=segmg.MG_F64, levels=1 if min(shape) < 4 else 2, sigma_blur=sigma,
                      model=model)
    o = O.Solver(img, mk, oracle_params(n, m, p))
    s.begin_step(); o.begin_step()
    for f in ("w", "z", "d"):
        assert relmax(s.level(0, f).cpu().numpy(), o.level(0, f)) < 1e-13, f
    assert relmax(s.phi().cpu().numpy(), o.phi) < 1e-13
    F = s.level(0, "F").cpu().numpy() - s.phi().cpu().numpy() / p.tau
    assert relmax(F, o.level(0, "Fn")) < 1e-12
    assert np.array_equal(s.mask().cpu().numpy() > 0, s.phi().cpu().numpy() > 0)
    s.close(); o.close()
