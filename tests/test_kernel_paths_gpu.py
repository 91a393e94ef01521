"""Kernels whose variant depends on size, type or boundary, at the sizes where the rule or the tiling
can go wrong, against the FP64 oracle or the general path."""
import numpy as np
import pytest

import oracle as O
from paper_2104_00095_gb300 import rmt, scenes as S
from parity_util import compare_state, needs_gpu, pair, rel_l2

pytestmark = [pytest.mark.gpu, needs_gpu]


def _box(n, periodic):
    """A flow without bodies on an n[0] x n[1] x n[2] grid: a lid between walls, or a smooth field
    in a periodic box; varying density needs no body here (the coefficient is 1)."""
    sc = S._box(max(n), periodic=periodic, lid=0.0 if periodic else 1.0)
    sc.update(n=tuple(n), hi=tuple(v / max(n) for v in n), mu=0.02)
    return sc


def _with_body(n, periodic):
    sc = _box(n, periodic)
    c = [0.5 * v / max(n) for v in n]
    r = 0.28 * min(n) / max(n)
    sc["solids"] = [S.solid(S.ELLIPSOID, c, (r, 0.8 * r, 0.9 * r), S.random_rotation(np.random.default_rng(2)),
                            rho_s=1.6, G=0.3, mu_a=0.02)]
    return sc


# coarsest levels of one block (3^3, 9 x 7 x 5, 11^3) and of a cluster with 1, 4 and 8 unknowns per
# thread (17 x 15 x 19, 23^3, 27^3), with walls and periodic; 54^3 = 2 x 27^3
@pytest.mark.parametrize("n,periodic", [((24, 24, 24), True), ((36, 28, 20), False), ((44, 44, 44), False),
                                        ((34, 30, 38), False), ((34, 38, 30), True), ((46, 46, 46), True),
                                        ((54, 54, 54), False)])
def test_coarsest_level_solves_fp64(n, periodic):
    """One step from a moving state, solved to 1e-13, against the oracle's conjugate gradients."""
    g, o = pair(_with_body(n, periodic))
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    g.write(rmt.RMT_F_U, u)
    assert o.write(O.F_U, u) == 0
    g.step(1)
    assert o.step(1) == 0, o.error()
    assert max(g.cycles()) <= 40  # the V-cycle keeps its rate only with an accurate coarsest solve
    compare_state(g, o, 1, 1e-10, tag=f"{n}")


@pytest.mark.parametrize("n,periodic", [((48, 48, 48), True), ((34, 30, 38), False), ((46, 46, 46), True),
                                        ((54, 54, 54), False)])
def test_coarsest_level_solves_fp32(n, periodic):
    """The FP32 form's adaptive solves to 1e-9 take about the cycles of the FP64 form's to 1e-9, and
    reach its velocities to FP32 accuracy."""
    out = []
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    for prec in ("fp64", "fp32"):
        g = rmt.Grid(dict(_with_body(n, periodic), precision=prec, mg_rtol=1e-9, mg_max_cycles=60))
        g.write(rmt.RMT_F_U, u)
        g.step(1)
        out.append((g.read(rmt.RMT_F_U), g.cycles()))
        g.close()
    (u64, c64), (u32, c32) = out
    assert rel_l2(u32, u64) <= 1e-5
    assert all(abs(a - b) <= 3 for a, b in zip(c64, c32)), (c64, c32)


@pytest.mark.parametrize("n", [(17, 15, 16), (23, 23, 23), (9, 7, 5)])
@pytest.mark.parametrize("ratio", [0.001, 0.01, 100.0, 1000.0])
def test_one_level_solves_at_density_ratios_fp64(n, ratio):
    """Grids of one level (an odd side) with a body far lighter or heavier than the fluid, solved to 1e-12.  Restated
    on the CPU, a solve leaves at most 2.7e-3 of its right-hand side at these ratios, so five gain twelve digits; one that
    left when a pass no longer halved the residual kept 0.3 to 0.5 of it at a ratio of 1/1000 and took above twenty."""
    sc = _with_body(n, False)
    sc["solids"][0]["rho_s"] = ratio
    sc.update(mg_rtol=1e-12, mg_max_cycles=60)
    g = rmt.Grid(sc)
    g.write(rmt.RMT_F_U, 0.1 * np.sin(np.arange(3 * np.prod(n)) * 0.37))
    g.step(1)
    assert max(g.cycles()) <= 8, g.cycles()
    g.close()


@pytest.mark.parametrize("n,periodic,precision", [((36, 40, 44), True, "fp32"), ((33, 35, 50), False, "fp32"),
                                                  ((36, 40, 44), True, "fp64")])
def test_float_reads_of_every_field(n, periodic, precision):
    """Float reads to the host, to device memory and to a device address that is not aligned to a
    float equal the rounded FP64 read; a reference map's is within one unit in the last place."""
    import torch

    g = rmt.Grid(dict(_with_body(n, periodic), precision=precision, mg_rtol=1e-6))
    g.write(rmt.RMT_F_U, 0.1 * np.sin(np.arange(3 * np.prod(n)) * 0.37))
    g.step(1)
    for f in list(range(1, 7)) + list(range(20, 35)):
        ref = g.read(f).astype(np.float32)
        raw = torch.zeros(ref.size * 4 + 8, dtype=torch.uint8, device="cuda")
        got = [g.read_float(f)]
        for off in (0, 2):
            g.read_float_ptr(f, raw.data_ptr() + off, ref.size * 4, 1)
            got.append(raw.cpu().numpy()[off:off + 4 * ref.size].copy().view(np.float32))
        for v in got:
            assert np.array_equal(np.isnan(v), np.isnan(ref)), f
            ok = ~np.isnan(ref)
            assert np.all(np.abs(v[ok] - ref[ok]) <= (np.spacing(np.abs(ref[ok])) if f in (4, 30) else 0)), f
    g.close()


@pytest.mark.parametrize("n,periodic", [((100, 98, 96), True), ((100, 74, 66), False)])
def test_float_reads_of_a_map_are_the_rounded_fp64_reads(n, periodic):
    """Every value of a body whose cell centres, from a corner at -0.3 in steps of 0.01, are not floats (of some 10^3
    displacements one makes a sum of a two-float centre round the other way)."""
    sc = dict(_with_body(n, periodic), precision="fp32", mg_rtol=1e-6, lo=(-0.3,) * 3)
    sc["hi"] = tuple(v / 100 - 0.3 for v in n)
    sc["solids"][0]["center"] = tuple(v - 0.3 for v in sc["solids"][0]["center"])
    g = rmt.Grid(sc)
    z, y, x = np.meshgrid(*[(np.arange(v) + 0.5) / 100 - 0.3 for v in n[::-1]], indexing="ij")
    for seed in range(4):
        w = np.random.default_rng(seed).uniform(5, 9, 3)
        xi = np.stack([c + 0.02 * np.sin(f * (x + 2 * y - z)) for c, f in zip((x, y, z), w)])
        g.write(rmt.RMT_F_XI, xi.reshape(-1))
        a, b = g.read_float(rmt.RMT_F_XI), g.read(rmt.RMT_F_XI).astype(np.float32)
        assert np.array_equal(a, b, equal_nan=True), np.count_nonzero((a != b) & ~np.isnan(b))
    g.close()


@pytest.mark.parametrize("layers,periodic,precision", [(1, True, "fp64"), (4, False, "fp64"), (8, True, "fp64"),
                                                       (4, True, "fp32")])
def test_extrapolation_of_unequal_bodies(layers, periodic, precision):
    """Bodies of unequal size extrapolated together: one across the seam, a small one, and a needle whose tip is
    a single line of cells, where the fits of radius 2 and 3 are degenerate and a wider search is taken."""
    n = (36, 28, 30)
    sc = _box(n, periodic)
    at = lambda i, j, k: tuple((v + 0.5) / max(n) for v in (i, j, k))
    size = lambda *r: tuple(v / max(n) for v in r)
    turn = S.random_rotation(np.random.default_rng(3))
    edge = at(1.3, 20.2, 27.9) if periodic else at(8.3, 19.2, 21.9)
    sc.update(band_layers=layers, precision=precision)
    sc["solids"] = [S.solid(S.ELLIPSOID, edge, size(6.4, 5.2, 4.3), turn, rho_s=1.4, G=0.2, mu_a=0.02),
                    S.solid(S.ELLIPSOID, at(18, 8, 8), size(7.6, 1.3, 1.3), rho_s=1.2, G=0.2, mu_a=0.02),
                    S.solid(S.SPHERE, at(27.6, 19.4, 14.7), size(2.6, 2.6, 2.6), rho_s=1.6, G=0.2, mu_a=0.02)]
    if precision == "fp32":
        sc.update(mg_rtol=1e-9, mg_max_cycles=60)
    g, o = pair(sc)
    u = 0.1 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    g.write(rmt.RMT_F_U, u)
    assert o.write(O.F_U, u) == 0
    g.step(2)
    assert o.step(2) == 0, o.error()
    if precision == "fp64":
        compare_state(g, o, 3, 1e-9)
    else:
        for m in range(3):
            assert np.array_equal(g.read(rmt.RMT_F_LAYER, m), o.read(O.F_LAYER, m))
            assert rel_l2(g.read(rmt.RMT_F_XI, m), o.read(O.F_XI, m)) <= 1e-5
    g.close()


def test_extrapolation_rounds_no_more_than_with_divisions():
    """Affine maps, which the fits reproduce but for rounding: the rms error of layers 1 and 3 over four bodies, in
    units of 2^-53.  Fits that divide have 5.16 and 6.91 of them, fits that multiply by a rounded reciprocal pivot 5.62 and
    7.77: the bounds lie midway."""
    import ctypes as C

    import torch

    wide, rms = np.longdouble, []
    for n, layers, r, seed in ((61, 5, 0.3, 1), (47, 4, 0.18, 4), (80, 5, 0.22, 5), (33, 3, 0.2, 2)):
        rng = np.random.default_rng(seed)
        sc = S._box(n, periodic=False)
        sc["band_layers"] = layers
        body = S.solid(S.ELLIPSOID, 0.5 + rng.uniform(-0.05, 0.05, 3), r * rng.uniform(0.6, 1.0, 3), S.random_rotation(rng))
        x = (np.arange(n) + 0.5) / n
        z, y, x = (v.reshape(-1).astype(wide) for v in np.meshgrid(x, x, x, indexing="ij"))
        m = np.eye(3) + 0.02 * rng.normal(size=(3, 3))
        exact = [wide(a) * x + wide(b) * y + wide(c) * z for a, b, c in m]
        xi = torch.tensor(np.stack([v.astype(np.float64) for v in exact])).cuda()
        out, phi = torch.empty_like(xi), torch.empty(n**3, dtype=torch.float64, device="cuda")
        lay = torch.empty(n**3, dtype=torch.int8, device="cuda")
        d, b = rmt.make_grid_desc(sc), rmt.make_solid_desc(body)
        assert rmt.load().rmt_extrapolate_noalloc(C.byref(d), C.byref(b), xi.data_ptr(), out.data_ptr(), phi.data_ptr(),
                                                  lay.data_ptr(), torch.cuda.current_stream().cuda_stream) == rmt.RMT_OK
        lay, out = lay.cpu().numpy(), out.cpu().numpy()
        err = lambda l: np.concatenate([(out[a][lay == l].astype(wide) - exact[a][lay == l]) for a in range(3)])
        rms.append([np.sqrt(np.mean(err(l).astype(np.float64)**2)) * 2.0**53 for l in (1, 3)])
    got = np.mean(rms, axis=0)
    assert got[0] <= 5.39 and got[1] <= 7.34, got


@pytest.mark.parametrize("n,periodic,precision", [((30, 12, 20), True, "fp32"), ((31, 13, 9), False, "fp32"),
                                                  ((62, 8, 44), True, "fp32"), ((4, 5, 6), False, "fp32"),
                                                  ((59, 6, 8), False, "fp32"), ((33, 9, 17), False, "fp64")])
def test_godunov_states_at_tile_edges(n, periodic, precision):
    """Face states where tiles of 30 x 6 columns end at, before and after the grid's last faces, against the
    oracle's (FP32 after one step from the same fields: rounding of the fields and of some hundred operations)."""
    sc = _box(n, periodic)
    sc.update(precision=precision)
    if precision == "fp32":
        sc.update(mg_rtol=1e-6, mg_max_cycles=60)
    g, o = pair(sc)
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    g.write(rmt.RMT_F_U, u)
    assert o.write(O.F_U, u) == 0
    g.step(1)
    assert o.step(1) == 0, o.error()
    for f, of in ((rmt.RMT_F_UFACE_X, O.F_UFACE_X), (rmt.RMT_F_UFACE_Y, O.F_UFACE_Y), (rmt.RMT_F_UFACE_Z, O.F_UFACE_Z)):
        assert rel_l2(g.read(f), o.read(of)) <= (1e-12 if precision == "fp64" else 1e-5)
    g.close()


@pytest.mark.parametrize("n", [(32, 30, 34), (33, 30, 32), (64, 40, 36), (34, 62, 30), (47, 33, 39)])
def test_fe_solve_with_walls_fp32(n):
    """Walled FE levels whose rows end at, before and after the last block's columns and begin at every alignment:
    the FP32 form's solves take the cycles of the FP64 form's and reach its velocities to FP32 accuracy."""
    out = []
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    for prec in ("fp64", "fp32"):
        g = rmt.Grid(dict(_box(n, False), precision=prec, mg_rtol=1e-9, mg_max_cycles=60))
        g.write(rmt.RMT_F_U, u)
        g.step(1)
        out.append((g.read(rmt.RMT_F_U), g.cycles()))
        g.close()
    (u64, c64), (u32, c32) = out
    assert rel_l2(u32, u64) <= 1e-5
    assert all(abs(a - b) <= 3 for a, b in zip(c64, c32)), (c64, c32)


@pytest.mark.parametrize("n,periodic", [((32, 32, 16), True), ((24, 20, 28), False), ((32, 16, 16), False),
                                        ((28, 32, 12), True), ((36, 32, 16), False),
                                        ((32, 32, 32), True), ((36, 32, 28), False)])
def test_small_mac_levels_in_one_block(n, periodic):
    """Levels of one block's cells (16 x 16 x 8 and 16 x 8 x 8 fill it in FP32 and FP64, 18 x 16 x 8 and 16^3 do not
    fit, odd rows): FP64 against the oracle, FP32 in the cycles of FP64 and to FP32 accuracy, the fused sweep's included."""
    sc = _box(n, periodic)
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    g, o = pair(sc)
    g.write(rmt.RMT_F_U, u)
    assert o.write(O.F_U, u) == 0
    g.step(1)
    assert o.step(1) == 0, o.error()
    compare_state(g, o, 0, 1e-10, tag=f"{n}")
    g.close()
    out = []
    for prec, sweep in (("fp64", 0), ("fp32", 0), ("fp32", 2)):
        g = rmt.Grid(dict(sc, precision=prec, mg_rtol=1e-9, mg_max_cycles=60, options={"mac_sweep": sweep}))
        g.write(rmt.RMT_F_U, u)
        g.step(1)
        out.append((g.read(rmt.RMT_F_U), g.cycles()))
        g.close()
    for v, c in out[1:]:
        assert rel_l2(v, out[0][0]) <= 1e-5
        assert all(abs(a - b) <= 3 for a, b in zip(out[0][1], c)), (out[0][1], c)


@pytest.mark.parametrize("shape,size,turn,precision", [(S.SPHERE, (8, 8, 8), False, "fp64"),
                                                       (S.ELLIPSOID, (8, 5, 3), False, "fp64"),
                                                       (S.ELLIPSOID, (11, 7.3, 2.2), True, "fp64"),
                                                       (S.ELLIPSOID, (11, 7.3, 2.2), True, "fp32"),
                                                       (S.SPHERE, (8.3, 8.3, 8.3), False, "fp32")])
def test_layer_zero_is_the_sign_of_the_level_set(shape, size, turn, precision):
    """Bodies whose surface passes through cell centres exactly (phi_0 = 0 there: not inside), and turned ones: the
    layers are the oracle's at every cell."""
    n = 32
    sc = S._box(n, periodic=False)
    sc.update(dt=0.2 / n, precision=precision)
    sc["solids"] = [S.solid(shape, (16.5 / n,) * 3, tuple(v / n for v in size),
                            S.random_rotation(np.random.default_rng(5)) if turn else None)]
    g, o = pair(sc)
    g.step(0)
    assert o.step(0) == 0, o.error()
    assert np.array_equal(g.read(rmt.RMT_F_LAYER, 0), o.read(O.F_LAYER, 0))
    g.close()


@pytest.mark.parametrize("n,precision,smooth", [((24, 20, 16), "fp32", 12.0), ((12, 12, 12), "fp32", 16.0),
                                                ((24, 20, 16), "fp64", 44.0), ((8, 8, 16), "fp64", 56.0)])
def test_profile_counts_the_bytes_of_the_kernels_that_run(n, precision, smooth):
    """Bytes per cell of a 7-point smoothing launch: a colour pass of x, the coefficient and half of b and x (FP32 one
    array, FP64 three and half the inverse diagonal), or a small level's sweeps in one block, every array once;
    the FP64 7-point residual's (x, b, three face arrays, r) and 27-point pass's (four stored arrays more)."""
    g = rmt.Grid(dict(_box(n, False), precision=precision, mg_rtol=1e-6))
    g.step(1)
    g.profile(True)
    g.step(1)
    g.profile(False)
    got = {p[0]: p[2:] for p in g.profile_read()}
    cells, nodes = np.prod(n), np.prod([v + 1 for v in n])
    names = list(got)
    assert got[names[13]][0] > 0 and got[names[13]][1] == smooth * cells
    if precision == "fp64":
        assert got[names[14]][1] == 48 * cells
        assert got[names[15]][1] == 56 * nodes + 8 * cells
    g.close()


@pytest.mark.parametrize("n,periodic", [((30, 28, 34), (0, 0, 0)), ((32, 36, 30), (0, 1, 0)), ((62, 30, 28), (0, 0, 1)),
                                        ((64, 28, 32), (0, 1, 1)), ((66, 30, 36), (0, 0, 0)), ((34, 28, 30), (1, 0, 0))])
def test_fe_tiles_of_two_levels_with_walls(n, periodic):
    """Even sides, so that the finest level is smoothed by the FE tiles: node rows that end before, at and after a block's
    last column (31, 33, 63, 65, 67), at every alignment, with periodic axes beside the walls.  FP64 against the oracle;
    FP32 in the cycles of FP64 and to FP32 accuracy."""
    assert all(v % 2 == 0 and v // 2 >= 3 for v in n)  # two levels at least
    sc = _box(n, False)
    sc["bc"] = [S.PERIODIC if periodic[d // 2] else S.NOSLIP for d in range(6)]
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    g, o = pair(sc)
    g.write(rmt.RMT_F_U, u)
    assert o.write(O.F_U, u) == 0
    g.step(1)
    assert o.step(1) == 0, o.error()
    compare_state(g, o, 0, 1e-10, tag=f"{n}")
    g.close()
    out = []
    for prec in ("fp64", "fp32"):
        g = rmt.Grid(dict(sc, precision=prec, mg_rtol=1e-9, mg_max_cycles=60))
        g.write(rmt.RMT_F_U, u)
        g.step(1)
        out.append((g.read(rmt.RMT_F_U), g.cycles()))
        g.close()
    (u64, c64), (u32, c32) = out
    assert rel_l2(u32, u64) <= 1e-5
    assert all(abs(a - b) <= 3 for a, b in zip(c64, c32)), (c64, c32)


@pytest.mark.parametrize("n,precision", [((90, 90, 10), "fp64"), ((58, 58, 58), "fp64"), ((70, 66, 66), "fp32")])
def test_coarsest_levels_beyond_a_cluster(n, precision):
    """Two-level grids whose coarsest level is solved by one block on global memory: 45 x 45 x 5 and 29^3 cells in FP64
    (their coefficients exceed a cluster's shared memory), 35 x 33 x 33 (more unknowns than a cluster holds)."""
    sc = _with_body(n, False)
    sc.update(precision=precision)
    u = 0.3 * np.sin(np.arange(3 * np.prod(n)) * 0.37)
    if precision == "fp64":
        g, o = pair(sc)
        g.write(rmt.RMT_F_U, u)
        assert o.write(O.F_U, u) == 0
        g.step(1)
        assert o.step(1) == 0, o.error()
        assert max(g.cycles()) <= 40
        compare_state(g, o, 1, 1e-10, tag=f"{n}")
    else:
        g = rmt.Grid(dict(sc, mg_rtol=1e-9, mg_max_cycles=60))
        g.write(rmt.RMT_F_U, u)
        g.step(1)
        assert max(g.cycles()) <= 40
    g.close()
