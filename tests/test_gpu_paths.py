"""The step's kernels at the sizes where their work splits change: tile edges
of the shell fill, the two sources of densities, the pair forces with and
without cell lists, the wide and the narrow coverage kernels, tile heights
and z chunks of the fused kernel, and captured single steps.

One step from random populations agrees with the FP64 oracle to 2e-6 on
populations of order 0.03 (a few FP32 ulps of the largest intermediate);
forces to 1e-5 of their largest (sums of FP32 link terms).  Where two splits of
the same work are compared, they agree bit for bit."""
import numpy as np
import pytest

from oracle import lbref
from paper_1109_3277_gb300 import lbe
from paper_1109_3277_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL_F, TOL_FORCE = 2e-6, 1e-5


def _one_step(shape, part, walls=False, mode="static", steps=1):
    """The library and the oracle after `steps` steps from random populations."""
    nx, ny, nz = shape
    f0 = W.random_populations(shape, seed=61)
    kw = dict(walls_z=walls, g_br=0.1)
    g = lbe.Lattice(shape, np.full((2, nz, ny, nx), 0.5), particle_mode=mode, **kw)
    r = lbref.Lattice(shape, np.full((2, nz, ny, nx), 0.5), particle_mode=lbe.MODES[mode], **kw)
    n = len(part["pos"])
    rp, ro, dr = (np.broadcast_to(part[k], (n,)).astype(float) for k in ("r_par", "r_perp", "delta_rho"))
    for L in (g, r):
        L.add_particles(part["pos"], part["quat"], rp, ro, dr, vel=part.get("vel"), omega=part.get("omega"))
        L.set_populations(f0)
        L.step(steps)
    return g, r


def _agree(g, r):
    _, _, tg = g.read_fields()
    _, _, tr = r.read_fields()
    assert np.array_equal(tg, tr)
    fl = tr == 0
    assert np.max(np.abs(g.get_populations()[:, :, fl] - r.get_populations()[:, :, fl])) < TOL_F
    pg, pr = g.read_particles(), r.read_particles()
    for k in ("force", "torque"):
        assert np.max(np.abs(pg[k] - pr[k])) < TOL_FORCE * max(1.0, np.abs(pr[k]).max()), k


# Boxes of one particle in tiles of 8 x 2 rows, with one and two tiles along x
# (30 nodes), and a box that is a whole period of the lattice; and one with so
# many tiles that they stay 10 x 5.
@pytest.mark.parametrize("shape,r_par,r_perp,tilt,rows", [((20, 22, 24), 2.3, 2.1, 0.3, (8, 2)),
                                                          ((24, 26, 40), 12.4, 3.2, 0.1, (8, 2)),
                                                          ((48, 24, 24), 13.6, 4.0, 1.5, (8, 2)),
                                                          ((44, 44, 44), 9.3, 8.7, 0.8, (8, 2)),
                                                          ((14, 30, 26), 5.2, 4.9, 1.1, (8, 2)),
                                                          ((48, 50, 46), 16.1, 6.3, 0.9, (10, 5))])
@pytest.mark.parametrize("walls", [False, True])
def test_shell_tiles_of_one_particle(shape, r_par, r_perp, tilt, rows, walls):
    part = dict(pos=[[shape[0] / 2 - 0.3, shape[1] / 2 + 0.2, shape[2] / 2 + 0.1]],
                quat=[W.axis_tilt_quaternion(tilt, 0.4)], r_par=r_par, r_perp=r_perp, delta_rho=0.07,
                vel=[[0.01, -0.02, 0.005]], omega=[[0.003, 0.002, -0.004]])
    g, r = _one_step(shape, part, walls)
    assert g.shell_tiles()[:2] == rows
    _agree(g, r)


def _big_and_small(shape, big, count, r_small):
    """One particle (centre at the middle of the lattice) and `count` spheres on
    a grid clear of it."""
    c = np.array(shape) / 2 + np.array([-0.3, 0.2, 0.1])
    ax = [np.arange(4.2 + 0.1 * k, shape[k] - 3.9, 7.3) for k in range(3)]
    p = np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)
    d = np.abs(p - c)
    reach = np.array([max(big[:2])] * 2 + [big[2]]) + r_small + 3.0  # half extents of the big one
    p = p[np.any(d > reach, axis=1)]
    assert len(p) >= count
    p = p[(np.arange(count) * len(p)) // count]
    return np.vstack([c, p]), np.array([big[0]] + [r_small] * count), np.array([big[1]] + [r_small] * count)


# Tiles of 30 x 22 x 22 nodes from 304 tiles on, every particle having as many as
# the largest: a tilted disc of radius 26, whose faces put 1,198 shell nodes
# and as many fluid nodes next to them into one tile (lists of 1,024 at a
# time), and a sphere across three edges of the tiles; with the densities
# summed in place, and with the density pass (more of the small spheres).
@pytest.mark.parametrize("big,tilt,count,dense", [((2.2, 26.0, 5.0), 0.03, 16, False), ((2.2, 26.0, 5.0), 0.03, 80, True),
                                                  ((15.2, 14.6, 15.2), 0.7, 38, False),
                                                  ((15.2, 14.6, 15.2), 0.7, 110, True)])
def test_large_shell_tiles_across_edges(big, tilt, count, dense):
    shape = (64, 66, 68)
    pos, rp, ro = _big_and_small(shape, big, count, 1.6)
    quat = np.tile(W.axis_tilt_quaternion(tilt, 0.4), (len(pos), 1))
    part = dict(pos=pos, quat=quat, r_par=rp, r_perp=ro, delta_rho=0.07,
                vel=W.uniform(80, (len(pos), 3), lo=-0.02, hi=0.02), omega=W.uniform(81, (len(pos), 3), lo=-4e-3, hi=4e-3))
    g, r = _one_step(shape, part)
    y, z, tiles, by_pass = g.shell_tiles()
    assert (y, z, by_pass) == (22, 22, dense) and tiles >= 8
    if big[0] < 3:
        # the disc's shell nodes in its tile 0 <= x < 30, 22 <= y < 44 from the box's corner
        t = g.read_fields(rho=False, vel=False)[2] == 2
        near = np.zeros_like(t)
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    if 0 < abs(dx) + abs(dy) + abs(dz) < 3:
                        near |= ~np.roll(t, (dz, dy, dx), (0, 1, 2))
        mid = [int(v) for v in np.round(pos[0])]
        lo = [int(np.floor(pos[0][k] - 26.0)) - 1 for k in range(2)]
        assert (t & near)[mid[2] - 5:mid[2] + 6, lo[1] + 22:lo[1] + 44, lo[0]:lo[0] + 30].sum() > 1024
    _agree(g, r)


# 5 small particles take tiles of 8 x 2 rows and sum their densities in place,
# 40 tiles of 10 x 5; from 255 on the density pass runs; 320 take tiles of 22 x
# 22 (link groups of 32) and the 128-thread coverage; 255 to 257 straddle the
# cell lists' threshold.
@pytest.mark.parametrize("count,rows,dense", [(5, (8, 2), False), (40, (10, 5), False), (255, (10, 5), True),
                                              (256, (10, 5), True), (257, (10, 5), True), (320, (22, 22), True)])
def test_many_particles_one_step(count, rows, dense):
    shape = (56, 52, 50)
    pos, quat = W.place_ellipsoids(shape, count, 3.0, 1.5, seed=62, margin=0.6)
    assert len(pos) == count
    part = dict(pos=pos, quat=quat, r_par=3.0, r_perp=1.5, delta_rho=-0.05,
                vel=W.uniform(63, (count, 3), lo=-2e-3, hi=2e-3), omega=W.uniform(64, (count, 3), lo=-2e-3, hi=2e-3))
    g, r = _one_step(shape, part, mode="free")
    tiles = g.shell_tiles()
    assert (tiles[:2], tiles[3]) == (rows, dense)
    _agree(g, r)


def test_dilute_suspension_in_large_tiles():
    """304 small spheres in a lattice they cover 1 % of: tiles of 22 x 22 rows
    with their densities summed in place."""
    shape, count = (82, 80, 78), 304
    pos, quat = W.place_ellipsoids(shape, count, 1.6, 1.6, seed=82, margin=0.8)
    assert len(pos) == count
    part = dict(pos=pos, quat=quat, r_par=1.6, r_perp=1.6, delta_rho=0.05,
                vel=W.uniform(83, (count, 3), lo=-2e-2, hi=2e-2), omega=W.uniform(84, (count, 3), lo=-2e-3, hi=2e-3))
    g, r = _one_step(shape, part)
    assert g.shell_tiles() == (22, 22, 1, False)
    _agree(g, r)


@pytest.mark.parametrize("count", [1, 151, 152])
def test_driven_particles_change_the_same_nodes(count):
    """Particles driven by up to 0.2 nodes a step for 8 steps: every covered
    and uncovered node is the oracle's, with 16 and with 4 warps a particle."""
    shape = (48, 46, 44)
    pos, quat = W.place_ellipsoids(shape, count, 3.0, 2.0, seed=65, margin=1.0)
    part = dict(pos=pos, quat=quat, r_par=3.0, r_perp=2.0, delta_rho=0.0,
                vel=W.uniform(66, (len(pos), 3), lo=-0.2, hi=0.2), omega=W.uniform(67, (len(pos), 3), lo=-0.05, hi=0.05))
    assert len(pos) == count
    g, r = _one_step(shape, part, mode="prescribed", steps=8)
    assert np.array_equal(g.read_fields()[2], r.read_fields()[2])


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("shape,walls,count", [((64, 20, 18), False, 0), ((64, 20, 18), True, 0), ((45, 20, 18), False, 0),
                                               ((64, 36, 30), False, 2), ((64, 36, 30), False, 20)])
def test_tiles_and_chunks_give_identical_results(shape, walls, count, storage):
    """Tile heights and z chunks (1 to beyond the lattice) split the same work:
    with and without solid nodes, tensor copies (nx = 45: none at 16 bit), and
    the density pass (20 particles)."""
    pos, quat = W.place_ellipsoids(shape, count, 4.0, 3.0, seed=68)
    out = []
    for rows, zc in ((None, 0), (8, 1), (8, 7), (4, 2), (4, 100)):
        nx, ny, nz = shape
        g = lbe.Lattice(shape, W.random_phases(shape, 0.5, seed=69), walls_z=walls, g_br=0.1, storage=storage)
        if count:
            g.add_particles(pos, quat, 4.0, 3.0, 0.05)
        if rows:
            g.set_tile(rows, zc)
        g.step(7)
        out.append(g.get_populations())
    for f in out[1:]:
        assert np.array_equal(out[0], f)


@pytest.mark.parametrize("nz,walls,count,storage,thick", [(30, False, 0, "f16", 24), (30, True, 0, "f32", 24),
                                                          (30, False, 1, "bf16", 24), (64, False, 700, "f16", 62)])
def test_bands_of_tiles_give_identical_results(nz, walls, count, storage, thick):
    """Layers of chunks too large for L2 go in bands of tile rows (35 rows of 8
    nodes as 18 and 17, 70 of 4 in up to four bands), as thin chunks do in one;
    with ψ on chip and (700 particles) from memory."""
    shape = (200, 277, nz)
    pos, quat = W.place_ellipsoids(shape, count, 4.0, 3.0, seed=72)
    rho0 = W.random_phases(shape, 0.5, seed=73)
    out = []
    for rows, zc in ((8, 2), (8, thick), (4, thick)):
        g = lbe.Lattice(shape, rho0, walls_z=walls, g_br=0.1, storage=storage)
        if count:
            g.add_particles(pos, quat, 4.0, 3.0, 0.05)
        g.set_tile(rows, zc)
        g.step(3)
        out.append(g.get_populations())
        g.close()
    for f in out[1:]:
        assert np.array_equal(out[0], f)


@pytest.mark.parametrize("mode,count", [("free", 1), ("free", 30), ("static", 2)])
def test_single_steps_replayed_equal_pairs_of_steps(mode, count):
    """40 single steps (direct, then a captured graph) and 40 at once (captured
    pairs, with the pair forces and the owner map's reset on a branch)."""
    shape = (40, 36, 34)
    pos, quat = W.place_ellipsoids(shape, count, 3.0, 2.0, seed=70)
    a, b = [], []
    for steps, out in (([1] * 40, a), ([40], b)):
        g = lbe.Lattice(shape, W.random_phases(shape, 0.5, seed=71), g_br=0.1, particle_mode=mode)
        g.add_particles(pos, quat, 3.0, 2.0, 0.05, vel=np.full((count, 3), 0.004))
        for n in steps:
            g.step(n)
        out += [g.get_populations(), g.read_fields()[2]] + [g.read_particles()[k] for k in ("pos", "quat", "force")]
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
