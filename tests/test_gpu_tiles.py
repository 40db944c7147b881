"""The tile kernel (one and two steps per launch) against the row march: the same
node arithmetic in other places, so the same bits.  tile_rows > 0 asks for the
row march; tile_rows = 0 lets the engine choose, which on these sizes is a tile
shape."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    torch.cuda.set_device(0)
    import paper_1202_6130_gb300 as p
    p.load()
    return p


def _case(nx, ny, lattice=9):
    w = W.droplet_on_wall(nx=nx, ny=ny, R=max(2.0, min(nx, ny) / 3.0), seed=nx + ny, noise_amp=1e-4,
                          lattice=lattice, tau=0.8)
    w.u_wall = np.zeros((2, ny, nx))
    w.u_wall[0] = 0.01 * W.uniform(3, ny * nx, 0.0, 1.0).reshape(ny, nx)
    w.u_wall[1] = -0.005
    w.body_force = (1e-5, -2e-6)
    w.epsilon = 1.3
    return w


def _run(pkg, w, storage, tile_rows, steps, **kw):
    sim = pkg.Simulation.from_workload(w, storage=storage, tile_rows=tile_rows, **kw)
    for n in steps:
        sim.step(n)
    f, clock = sim.populations(), sim.clock()
    sim.close()
    return f, clock


# D2Q9: smaller than a halo, than a tile, one more and one less than tiles of 32
# and 64 columns and 4, 8, 12 and 24 rows, odd widths (one step per launch, a
# lone last column), and the sizes from which the larger shapes are chosen.
D2Q9 = [(1, 1), (2, 3), (4, 4), (6, 5), (8, 256), (32, 8), (34, 9), (62, 7), (64, 12), (66, 13),
        (67, 35), (130, 25), (254, 49), (512, 384), (1026, 515), (1537, 771), (2048, 1024)]


@pytest.mark.parametrize("size", D2Q9, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("storage", ["fp32", "fp16s", "bf16s"])
def test_tiles_equal_the_row_march_bitwise(pkg, size, storage):
    """Seven steps (three launches of two and one of one, or seven of one), then
    one and four more."""
    w = _case(*size)
    want, c0 = _run(pkg, w, storage, 3, (7, 1, 4))
    got, c1 = _run(pkg, w, storage, 0, (7, 1, 4))
    np.testing.assert_array_equal(got, want)
    assert c0 == c1


@pytest.mark.parametrize("kw", [dict(rounding="nearest"), dict(project=True)],
                         ids=["nearest", "project"])
@pytest.mark.parametrize("storage", ["fp32", "bf16s"])
def test_tiles_equal_the_row_march_with_run_time_switches(pkg, storage, kw):
    w = _case(130, 50)
    for size in ((130, 50), (1026, 515)):
        w = _case(*size)
        np.testing.assert_array_equal(_run(pkg, w, storage, 0, (6,), **kw)[0],
                                      _run(pkg, w, storage, 4, (6,), **kw)[0])


@pytest.mark.parametrize("size", [(1, 1), (5, 2), (17, 9), (33, 29), (66, 17), (131, 40), (1026, 515)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("lattice,storage", [(9, "fp64"), (21, "fp64"), (21, "fp32"), (21, "fp16s"),
                                             (21, "bf16s")])
def test_one_step_tiles_equal_the_row_march_bitwise(pkg, lattice, storage, size):
    w = _case(*size, lattice=lattice)
    np.testing.assert_array_equal(_run(pkg, w, storage, 0, (3,))[0], _run(pkg, w, storage, 4, (3,))[0])


def test_more_tile_rows_than_a_grid_holds(pkg):
    """270,000 rows: 67,500 tiles of 4 rows in one column, beyond a grid's 65,535
    in y.  The read-out (tiles of 4 rows) and two steps equal the row march."""
    nx, ny = 8, 270000
    rho = 1.0 + 0.1 * W.uniform(5, nx * ny, -1.0, 1.0).reshape(ny, nx)
    out = []
    for tile_rows in (0, 8):
        sim = pkg.Simulation(nx, ny, storage="fp16s", tile_rows=tile_rows, shift_rho=1.0)
        sim.set_equilibrium(rho)
        r0 = sim.moments()[0]
        assert np.abs(r0 - rho).max() < 1e-3
        sim.step(3)
        out.append(sim.populations())
        sim.close()
    np.testing.assert_array_equal(out[0], out[1])


def test_checks_fall_between_the_steps_of_two(pkg):
    """check_every = 3 reports a non-finite density on the step it is due (the
    state stays as after that step), although two steps fit one launch."""
    w = _case(64, 32)
    sim = pkg.Simulation.from_workload(w, storage="fp32", check_every=3)
    f = sim.populations()
    f[:, 10, 10] = np.nan
    sim.set_populations(f)
    with pytest.raises(pkg.LbmError) as ei:
        sim.step(8)
    assert "ENONFINITE" in str(ei.value) and sim.steps_done() == 3
    sim.close()


def test_fp64_psi_scale_other_than_one_matches_oracle(pkg):
    """rho0 = 0.7: the FP64 quotient rho / rho0 by reciprocal and remainder."""
    from oracle import lbm_oracle as O
    w = _case(45, 26)
    w.rho0 = 0.7
    p = O.Params(lattice=O.D2Q9, tau=w.tau, G=w.G, rho0=w.rho0, body_force=tuple(w.body_force))
    wall = O.Wall(w.phi_s, w.psi_r, w.psi_a, w.G_R, w.G_A, w.epsilon, w.u_wall)
    f = O.run(p, wall, O.initial_populations(p, w.rho, w.ux, w.uy, w.noise), 20)
    got, _ = _run(pkg, w, "fp64", 0, (20,))
    np.testing.assert_allclose(got, f, rtol=1e-12, atol=1e-15)


def test_fp32_velocity_quotient_is_within_an_ulp_of_fp64(pkg):
    """Without forces u = j / rho, j and rho formed in FP32 from the populations
    as the kernel forms them: the read-out's quotient of FP32 numbers differs
    from the FP64 division by at most one unit in the last place (2^-52
    relative), for ordinary, tiny (down to 1e-25: the division itself), zero
    and negative momenta."""
    ny, nx = 64, 66
    rng = np.random.default_rng(5)
    f = rng.uniform(0.01, 0.5, (9, ny, nx)).astype(np.float32)
    scale = 10.0 ** rng.uniform(-25, 0, (ny, nx)).astype(np.float32)
    f[1:, ::2] = (rng.standard_normal((8, ny, nx)) * scale).astype(np.float32)[:, ::2]
    f[5, ::4] = f[7, ::4] = f[6, ::4] = f[8, ::4] = 0.25
    f[1, ::4] = f[3, ::4]                                      # j_x = 0
    sim = pkg.Simulation(nx, ny, storage="fp32", G=0.0)
    sim.set_populations(f.astype(np.float64))
    rho, ux, uy = sim.moments()
    r = f[0].copy()
    for i in range(1, 9):
        r = r + f[i]
    d57, d86 = f[5] - f[7], f[8] - f[6]
    jx = ((f[1] - f[3]) + d57) + d86
    jy = ((f[2] - f[4]) + d57) - d86
    np.testing.assert_array_equal(rho, r.astype(np.float64))
    for u, j in ((ux, jx), (uy, jy)):
        want = j.astype(np.float64) / r.astype(np.float64)
        assert (np.abs(u - want) <= 2.0 ** -52 * np.abs(want)).all()
    sim.close()


def test_fp32_velocity_quotient_at_any_density(pkg):
    """The same for densities from 2^-44 to 2^44 and momenta down to FP32's
    subnormal numbers (quotients whose words leave FP32's normal range are
    divided in FP64), and for a momentum of zero under a subnormal force."""
    ny, nx = 128, 128
    rng = np.random.default_rng(11)
    f = np.zeros((9, ny, nx), np.float32)
    f[0] = np.ldexp(rng.uniform(1.0, 2.0, (ny, nx)), rng.integers(-44, 44, (ny, nx)))
    for i, j in ((1, 3), (2, 4)):  # j_x and j_y to three words: f1 - f3 is rounded once
        f[i] = np.ldexp(rng.uniform(-2.0, 2.0, (ny, nx)), rng.integers(-148, -44, (ny, nx)))
        f[j] = f[i] * rng.uniform(0.0, 1.0, (ny, nx)).astype(np.float32)
    f[1:5, ::8] = 0.0
    for body in (0.0, 2.0 ** -149):
        sim = pkg.Simulation(nx, ny, storage="fp32", G=0.0, body_force=(body, body))
        sim.set_populations(f.astype(np.float64))
        rho, ux, uy = sim.moments()
        r = f[0].copy()
        for i in range(1, 9):
            r = r + f[i]
        np.testing.assert_array_equal(rho, r.astype(np.float64))
        for u, j in ((ux, f[1] - f[3]), (uy, f[2] - f[4])):
            want = (j.astype(np.float64) + 0.5 * body) / r.astype(np.float64)
            assert (np.abs(u - want) <= 2.0 ** -52 * np.abs(want)).all()
        sim.close()


def test_fp64_velocity_where_the_density_is_zero_or_infinite(pkg):
    """u = j / rho as the FP64 division gives it: infinite or not a number at
    rho = 0, zero at an infinite rho, and ordinary elsewhere."""
    ny, nx = 6, 16
    f = np.full((9, ny, nx), 0.1)
    f[1] = 0.25                                    # j_x = 0.15
    f[:, 2, 3], f[1, 2, 3], f[0, 2, 3] = 0.0, 0.25, -0.25      # rho = 0, j = (0.25, 0)
    f[:, 4, 9] = 0.0                                           # rho = 0, j = 0
    f[0, 1, 5] = np.inf                                        # rho infinite, j finite
    sim = pkg.Simulation(nx, ny, storage="fp64", G=0.0)
    sim.set_populations(f)
    rho, ux, uy = (a.cpu().numpy() for a in sim.moments_device())
    sim.close()
    r = f.sum(0)
    assert rho[2, 3] == 0.0 and rho[4, 9] == 0.0 and rho[1, 5] == np.inf
    assert ux[2, 3] == np.inf and np.isnan(uy[2, 3])
    assert np.isnan(ux[4, 9]) and np.isnan(uy[4, 9])
    assert ux[1, 5] == 0.0 and uy[1, 5] == 0.0
    ok = np.isfinite(r) & (r != 0.0)
    np.testing.assert_allclose(ux[ok], 0.15 / r[ok], rtol=1e-13)


# A size that selects each tile shape of a (lattice, storage), with remainders in x
# and y (odd widths where one-step D2Q9 shapes are to run), and the sizes at which
# the two-step shapes run in practice.
SHAPES = {
    (9, "fp64"): {(16, 4, 1): [(49, 9)], (32, 8, 1): [(1457, 17), (2049, 259)],
                  (32, 16, 1): [(193, 1267), (520, 500)]},
    (21, "fp64"): {(16, 4, 1): [(49, 9)], (32, 8, 1): [(1459, 17)], (32, 16, 1): [(97, 435), (333, 203)]},
    (21, "fp32"): {(16, 4, 1): [(49, 9)], (32, 8, 1): [(1258, 17), (651, 150)],
                   (64, 8, 1): [(10769, 58), (1250, 500)]},
    (21, "fp16s"): {(32, 4, 1): [(97, 9), (651, 150)], (64, 8, 1): [(418, 1510), (1250, 300)]},
    (9, "fp32"): {(32, 4, 1): [(97, 9)], (64, 8, 1): [(6753, 21), (1537, 771)], (32, 4, 2): [(98, 9)],
                  (32, 8, 2): [(134, 927), (402, 203)], (32, 28, 2): [(520, 1502), (1538, 771)],
                  (64, 12, 2): [(5236, 33), (1026, 515)], (64, 22, 2): [(11064, 61), (2050, 1027)]},
    (9, "fp16s"): {(32, 4, 1): [(97, 9)], (64, 8, 1): [(289, 1339), (1538, 771)], (32, 4, 2): [(98, 9)],
                   (32, 8, 2): [(130, 739), (400, 201)], (32, 28, 2): [(130, 1526), (1026, 515)],
                   (64, 12, 2): [(6910, 33)], (64, 22, 2): [(6606, 65), (12160, 41)]},
}
SHAPES[9, "bf16s"], SHAPES[21, "bf16s"] = SHAPES[9, "fp16s"], SHAPES[21, "fp16s"]
SHAPE_CASES = [(q, st, shape, size) for (q, st), shapes in SHAPES.items()
               for shape, sizes in shapes.items() for size in sizes]


@pytest.mark.parametrize("lattice,storage,shape,size", SHAPE_CASES,
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_each_tile_shape_equals_the_row_march_bitwise(pkg, lattice, storage, shape, size):
    """The shape that runs is the one meant (columns, rows and steps of a launch,
    from the layout), and four steps and one more give the row march's bits."""
    w = _case(*size, lattice=lattice)
    sim = pkg.Simulation.from_workload(w, storage=storage)
    lay = sim.layout()
    bytes_per_step = 2 * lattice * {"fp64": 8, "fp32": 4}.get(storage, 2)
    assert lay["stages"] == 1
    assert (lay["strip_width"], lay["tile_rows"], bytes_per_step // lay["bytes_per_node"]) == shape
    sim.step(4)
    sim.step(1)
    march = pkg.Simulation.from_workload(w, storage=storage, tile_rows=4)
    assert march.layout()["stages"] > 1
    march.step(5)
    np.testing.assert_array_equal(sim.populations(), march.populations())
    sim.close()
    march.close()


@pytest.mark.parametrize("lattice,storage,size", [(9, "fp64", (520, 500)), (21, "fp64", (333, 203)),
                                                  (21, "fp32", (1250, 500)), (21, "bf16s", (1250, 300)),
                                                  (9, "fp32", (1537, 771)), (9, "fp16s", (1026, 515))],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_shapes_with_inner_tiles_equal_the_row_march_with_run_time_switches(pkg, lattice, storage, size):
    """The equation-of-state psi and the projection, on lattices with tiles that run
    the copy of the update without edges and walls."""
    w = _case(*size, lattice=lattice)
    w.psi_kind, w.G = 1, -1.0
    want = _run(pkg, w, storage, 4, (5,), project=True)[0]
    assert np.isfinite(want).all()
    np.testing.assert_array_equal(_run(pkg, w, storage, 0, (4, 1), project=True)[0], want)


def test_full_size_two_step_tiles_match_oracle_and_the_row_march(pkg):
    """Two steps of the 8192x4096 multi-droplet lattice in one launch, as the
    benchmark takes them, after 20 steps: 70 sampled nodes (tile edges in x and y,
    wall rows, the periodic seam) recomputed by the oracle from a periodic 11x11
    window of the FP32 state (the reach of two steps is 4), within twice the
    bound of one step (1e-5); and every population equal to two row marches."""
    from oracle import lbm_oracle as O
    w = W.large_multi_droplet(noise_amp=1e-6)
    sim = pkg.Simulation.from_workload(w, storage="fp32")
    lay = sim.layout()
    tw, th = lay["strip_width"], lay["tile_rows"]
    assert lay["stages"] == 1 and lay["bytes_per_node"] == 36     # two steps per launch
    sim.step(20)
    f0 = sim.populations()
    sim.step(2)
    f2 = sim.populations()
    sim.close()
    march = pkg.Simulation.from_workload(w, storage="fp32", tile_rows=4)
    march.set_populations(f0)
    march.step(2)
    np.testing.assert_array_equal(f2, march.populations())
    march.close()
    p = O.Params(lattice=O.D2Q9, tau=w.tau, G=w.G, rho0=w.rho0, body_force=tuple(w.body_force))
    r = 5
    rng = np.random.default_rng(2)
    ys = list(rng.integers(0, w.ny, 40)) + [0, 1, 2, w.ny - 1, w.ny - 2, th - 1, th, th + 1, 2 * th - 1,
                                           2 * th] + [100 * th + d for d in range(-3, 7)]
    xs = list(rng.integers(0, w.nx, 40)) + [0, w.nx - 1, 1, tw - 1, tw, tw + 1, 2 * tw - 1, w.nx - tw,
                                           4095, 4096] + [50 * tw + d for d in range(-4, 6)]
    for y, x in zip(ys, xs):
        at = np.ix_(np.arange(y - r, y + r + 1) % w.ny, np.arange(x - r, x + r + 1) % w.nx)
        wall = O.Wall(w.phi_s[at], w.psi_r[at], w.psi_a[at], w.G_R, w.G_A, w.epsilon)
        fo = np.stack([f[at] for f in f0])
        for _ in range(2):
            fo = O.step(p, wall, fo)
        err = np.max(np.abs(f2[:, y, x] - fo[:, r, r]) / np.maximum(np.abs(fo[:, r, r]), 1e-3))
        assert err < 2e-5, (y, x, err)
