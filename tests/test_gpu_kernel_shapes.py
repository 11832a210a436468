"""Kernels whose tiles, chunks or algorithm depend on the grid, at the sizes where a
tile, a run or a chunk ends: GPU results against the FP64 oracle."""

import numpy as np
import pytest

import oracle
from test_gpu_parity import rel, setup_case

pytestmark = pytest.mark.gpu


# rows shorter and longer than a double-precision stress tile (8 .. 64 columns), heights
# that leave one row in the last tile, chunks of one plane and chunks with a remainder;
# the smallest grids wrap every stencil round the box
@pytest.mark.parametrize("shape", [(8, 4, 8, True), (8, 8, 8, False), (18, 7, 8, True), (36, 29, 9, True),
                                   (64, 9, 12, False), (72, 54, 16, False), (96, 17, 27, True), (162, 13, 8, True)])
@pytest.mark.parametrize("model,extra", [('oldroyd_b', {}), ('saramito', {'Bi': 0.4}), ('fene_p', {'L2': 60.0})])
def test_double_precision_stress_tiles(evp, shape, model, extra):
    import torch
    sim, st, g, prm = setup_case(evp, shape, model, extra, evp.EVP_FP64)
    out = torch.empty((6,) + sim.shape, dtype=torch.float64, device='cuda')
    evp.evp_stress_rhs(sim.handle, out)
    sim.sync()
    ref = oracle.stress_rhs(st.U, st.V, st.W, st.B, g, prm)
    for c in range(6):
        assert rel(out[c].cpu().numpy(), ref[c]) < 1e-12, (c, rel(out[c].cpu().numpy(), ref[c]))


# momentum tiles: 64 x 4 (nx a multiple of 64), 32 x 8, element-wise staging (nx % 4 = 2);
# the last tile row holding one row, the wall rows in one tile, chunks with a remainder;
# Newtonian states stage no stress
@pytest.mark.parametrize("shape", [(64, 4, 8, True), (64, 5, 27, True), (128, 9, 8, True), (32, 8, 9, True),
                                   (36, 17, 8, True), (18, 13, 16, True), (64, 18, 54, False), (54, 16, 8, False)])
@pytest.mark.parametrize("model", ['oldroyd_b', 'newtonian'])
@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-5)])
def test_momentum_tiles(evp, shape, model, prec, tol):
    sim, st, g, prm = setup_case(evp, shape, model, {}, prec, dpdx=0.3)
    # a quarter of the explicit viscous limit dt 4 mu_s sum 1/h^2 <= 2.51
    h2 = sum((n / l) ** 2 for n, l in zip(shape[:3], (g.lx, g.ly, g.lz)))
    dt = min(1e-3, 0.25 * 2.51 / (4 * 0.4 / 2.0 * h2))
    for _ in range(2):
        sim.step(dt)
        st = oracle.rk3_step(st, dt, g, prm, force=(0.3, 0.0, 0.0))
    sim.sync()
    for f, ref in ((evp.EVP_U, st.U), (evp.EVP_V, st.V), (evp.EVP_W, st.W)):
        assert rel(sim.get(f), ref) < tol, (f, rel(sim.get(f), ref))


# several fields to device buffers in one launch: whole and broken 16-byte words, buffers
# off the 16-byte grid, buffers that overlap (copied in order)
@pytest.mark.parametrize("shape", [(8, 4, 8, True), (18, 5, 9, True), (64, 32, 24, False)])
@pytest.mark.parametrize("prec", [0, 1])
def test_device_field_copies(evp, shape, prec):
    import torch
    sim, _, _, _ = setup_case(evp, shape, 'oldroyd_b', {}, prec)
    n = sim.shape[0] * sim.shape[1] * sim.shape[2]
    fields = [evp.EVP_U, evp.EVP_P, evp.EVP_BXY, evp.EVP_BZZ]
    want = [sim.get(f).ravel() for f in fields]
    for skew in (0, 1, 2):
        pool = torch.full((4 * (n + 8),), float('nan'), dtype=sim.dtype, device='cuda')
        bufs = [pool[q * (n + 8) + skew:q * (n + 8) + skew + n] for q in range(4)]
        evp.evp_get_fields(sim.handle, fields, bufs)
        for b, w in zip(bufs, want):
            assert np.array_equal(b.cpu().numpy(), w)
        assert int(torch.isnan(pool).sum()) == 32
    pool = torch.zeros(2 * n, dtype=sim.dtype, device='cuda')
    evp.evp_get_fields(sim.handle, fields[:2], [pool[:n], pool[n // 2:n // 2 + n]])
    assert np.array_equal(pool[n // 2:n // 2 + n].cpu().numpy(), want[1])
    assert np.array_equal(pool[:n // 2].cpu().numpy(), want[0][:n // 2])


# the single-precision monitoring filters where every cell is in doubt: a uniform B (all
# determinants and traces equal), a deviator exactly at the yield stress, tiny and huge
# values, an infinity; and a velocity at rest, uniform, and solenoidal to rounding
@pytest.mark.parametrize("shape", [(36, 9, 8, True), (64, 16, 24, False)])
@pytest.mark.parametrize("kind", ['uniform', 'yield', 'tiny', 'huge', 'inf'])
def test_single_precision_monitoring_filters(evp, shape, kind):
    from oracle import diagnostics as odg
    sim, st, g, prm = setup_case(evp, shape, 'saramito', {'Bi': 0.4}, evp.EVP_FP32)
    rng = np.random.default_rng(3)
    full = lambda v: np.full(sim.shape, v)
    B = {'uniform': lambda: [full(v) for v in (1.5, 0.25, 0.1, 1.2, 0.3, 1.1)],
         # |tau^d| of a pure shear B = I + b e_xy is (mu_p/lambda) b: at the yield stress to rounding
         'yield': lambda: [full(1.0), full(np.float32(0.4 / 2.0 * 0.8 / (0.6 / 2.0))), full(0.0), full(1.0), full(0.0), full(1.0)],
         'tiny': lambda: [rng.uniform(0.5, 2.0, sim.shape) * 1e-20 for _ in range(6)],
         'huge': lambda: [rng.uniform(0.5, 2.0, sim.shape) * 1e20 for _ in range(6)],
         'inf': lambda: [b.copy() for b in st.B]}[kind]()
    if kind == 'inf':
        B[3][1, 2, 3] = np.inf
    if kind in ('uniform', 'yield'):
        U, V, W = full(0.0 if kind == 'uniform' else 0.75), full(0.0), full(0.0)
    else:
        U, V, W = st.U, st.V, st.W
    sim.set_state(U, V, W, None, B)
    rd = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    with np.errstate(all='ignore'):
        ref = odg.diagnostics(rd(U), rd(V), rd(W), [rd(b) for b in B], g, prm)
    got = sim.diagnostics()
    for f in ('min_det_B', 'max_tr_B', 'yielded_cells', 'nonfinite_cells'):
        assert got[f] == ref[f], (f, got[f], ref[f])
    assert got['kinetic_energy'] == pytest.approx(ref['kinetic_energy'], rel=1e-12, abs=0)
    assert abs(got['max_div'] - ref['max_div']) <= 1e-12 * 2.0 / min(g.dx, g.dy, g.dz)


# level-set stages whose z chunks hold three planes and a remainder: advection by u^n and
# re-distancing of a field that repeats 32 times along z must repeat bit for bit, and be
# what one period gives on its own (a grid of one plane per chunk)
@pytest.mark.parametrize("nx,ny,walls", [(36, 113, True), (36, 128, False)])
@pytest.mark.parametrize("prec", [0, 1])
def test_level_set_chunks(evp, nx, ny, walls, prec):
    rng = np.random.default_rng(5)
    one = (8, ny, nx)
    k, j, i = np.meshgrid(*(np.arange(m) for m in one), indexing='ij')
    phi = 0.2 * np.cos(2 * np.pi * i / nx) + 0.1 * np.cos(np.pi * j / ny) + 0.05 * np.sin(2 * np.pi * k / 8)
    vel = [rng.uniform(-1, 1, one) for _ in range(3)]
    if walls:
        vel[1][:, -1] = 0.0
    prm = evp.make_params(Re=35.0, Wi=1.0, beta=0.5, precision=prec, integrator=evp.EVP_AB2, mu_ratio=1.0,
                          ls_eps_cells=1.5, sigma=0.1, drho_g=1.0, reinit_every=1, reinit_iters=2)
    got = []
    for reps in (1, 32):
        sim = evp.Simulation(evp.make_grid(nx, ny, 8 * reps, 1.0, 4.0, 0.25 * reps, walls), 'oldroyd_b', prm)
        sim.set_state(*(np.tile(v, (reps, 1, 1)) for v in vel))
        sim.set(evp.EVP_PHI, np.tile(phi, (reps, 1, 1)))
        sim.step(1e-3)
        sim.sync()
        got.append(sim.get(evp.EVP_PHI))
    assert np.isfinite(got[0]).all() and not np.array_equal(got[0], phi.astype(got[0].dtype))
    assert np.array_equal(got[1], np.tile(got[0], (32, 1, 1)))


# the trace limit of a B that is no longer positive definite: diagonals of 1e7 cancel to a
# trace 0.1 above or 0.3 below L^2, less than a single-precision rounding of theirs
@pytest.mark.parametrize("bzz,hit", [(59.7, True), (59.3, False)])
def test_double_precision_trace_limit_of_cancelling_diagonals(evp, bzz, hit):
    sim, st, g, prm = setup_case(evp, (36, 9, 8, True), 'fene_p', {'L2': 60.0}, evp.EVP_FP64)
    full = lambda v: np.full(sim.shape, v)
    sim.set_state(full(0.0), full(0.0), full(0.0), full(0.0),
                  [full(v) for v in (1e7 + 0.4, 0.0, 0.0, -1e7, 0.0, bzz)])
    sim.sync(raise_on_error=False)
    sim.step(1e-24)
    bits = sim.sync(raise_on_error=False)[1]
    assert bool(bits & evp.EVP_BIT_TRACE_LIMIT) == hit


# the closures where |tau^d|^2 overflows or is below the range of the refined reciprocal
# square root, and where tr B = L^2 exactly, of a uniform B at rest: RT = (a I - F B)/lambda
@pytest.mark.parametrize("model,extra,b,want", [
    ('saramito', {'Bi': 0.4}, (1e160, 0.0, 0.0, 1.0, 0.0, 1.0), ((1.0 - 1e160) / 0.8, 0.0, 0.0, 0.0, 0.0, 0.0)),   # F = 1
    ('saramito', {'Bi': 0.4}, (1.0, 1e-100, 0.0, 1.0, 0.0, 1.0), (0.0, 0.0, 0.0, 0.0, 0.0, 0.0)),                 # F = 0
    ('saramito', {'Bi': 0.0}, (1.0, 1e-100, 0.0, 1.0, 0.0, 1.0), (0.0, -1e-100 / 0.8, 0.0, 0.0, 0.0, 0.0)),       # F = 1
    ('fene_p', {'L2': 60.0}, (20.0, 1.0, 1.0, 20.0, 1.0, 20.0), (-np.inf,) * 6)])                                  # F = inf
def test_double_precision_closures_at_the_ends_of_the_range(evp, model, extra, b, want):
    import torch
    sim, _, _, _ = setup_case(evp, (36, 9, 8, True), model, extra, evp.EVP_FP64)
    z = np.zeros(sim.shape)
    sim.set_state(z, z, z, z, [z + v for v in b])
    out = torch.empty((6,) + sim.shape, dtype=torch.float64, device='cuda')
    evp.evp_stress_rhs(sim.handle, out)
    sim.sync(raise_on_error=False)
    for c in range(6):
        np.testing.assert_allclose(out[c].cpu().numpy(), z + want[c], rtol=1e-14, atol=0)


# chunks of three planes and more with a short last one, by the chunk rules themselves: 32 x
# 8 momentum tiles staged by element (nx % 4 = 2) and in 16-byte chunks, 64 x 4 tiles, walls
# (planes whose ghost rows are set inside the march) and none, the double-precision kernels
@pytest.mark.parametrize("shape,prec", [
    ((18, 33, 64, True), 1), ((36, 33, 32, True), 1), ((36, 36, 32, False), 1), ((64, 17, 64, True), 1),
    ((128, 33, 54, True), 1), ((18, 29, 64, True), 0), ((36, 33, 32, True), 0), ((72, 36, 54, False), 0)])
@pytest.mark.parametrize("model,extra", [('saramito', {'Bi': 0.4}), ('newtonian', {})])
def test_chunks_with_a_remainder(evp, shape, prec, model, extra):
    sim, st, g, prm = setup_case(evp, shape, model, extra, prec, dpdx=0.3)
    cfg = evp.evp_tile_config_get(sim.grid, prec, model)
    for kz in (cfg.stress_kz, cfg.momentum_kz):
        assert kz > 2 and shape[2] % kz, kz
    # a quarter of the explicit viscous limit dt 4 mu_s sum 1/h^2 <= 2.51
    h2 = sum((n / l) ** 2 for n, l in zip(shape[:3], (g.lx, g.ly, g.lz)))
    dt = min(1e-3, 0.25 * 2.51 / (4 * 0.4 / 2.0 * h2))
    for _ in range(2):
        sim.step(dt)
        st = oracle.rk3_step(st, dt, g, prm, force=(0.3, 0.0, 0.0))
    sim.sync()
    pairs = [(evp.EVP_U, st.U), (evp.EVP_V, st.V), (evp.EVP_W, st.W)]
    if model != 'newtonian':
        pairs += [(evp.EVP_BXX + c, st.B[c]) for c in range(6)]
    for f, ref in pairs:
        assert rel(sim.get(f), ref) < (1e-5 if prec else 1e-10), (f, rel(sim.get(f), ref))
