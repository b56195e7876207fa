"""Launch shapes at the sizes where they can differ (marked gpu): cells of 1 to over 100 particles
(hit masks of 32 candidates, aligned groups of four, two masks per lane), coincident particles,
lists cut at their last entry, particle counts around a warp: every build variant writes one list,
the oracle's sets, and every force shape the same bits."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2207_11328_gb300 import N_BUILD_VARIANTS, N_FORCES_VARIANTS, scenes
from tests.gpu_common import compare_neighbor_sets, launches, rel_check, require_gpu, sim_for

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


def _cloud(n, cells, crowd, periodic, n_boundary=0, seed=1):
    """n random particles in a box of cells^3 grid cells, `crowd` of them in one cell (at its
    corner), a few coincident; the last n_boundary are boundary particles."""
    rng = np.random.default_rng(seed)
    s = scenes.periodic_box(n_per_axis=4, dp=0.02)
    R = 2 * s.h
    L = cells * R * 1.01
    pos = rng.uniform(0, L, (n, 3))
    pos[:crowd] = rng.uniform(0.05 * R, 0.95 * R, (crowd, 3))
    if n > 3:
        pos[n // 2] = pos[0]  # coincident: no pair
    ptype = np.zeros(n, np.uint8)
    if n_boundary:
        ptype[n - n_boundary:] = 1
    vel = rng.uniform(-0.1, 0.1, (n, 3)).astype(np.float32)
    vel[ptype == 1] = 0
    return dataclasses.replace(s, pos=pos, vel=vel, delta=rng.uniform(-1e-3, 1e-3, n).astype(np.float32),
                               mass=np.full(n, 8e-3, np.float32), ptype=ptype, scene=np.zeros(n, np.uint32),
                               origin=(0.0, 0.0, 0.0), size=(L, L, L), periodic=7 if periodic else 0)


@pytest.mark.parametrize("n,cells,crowd,periodic,nb", [(1, 3, 0, True, 0), (31, 3, 0, False, 5), (33, 4, 29, True, 3),
                                                       (200, 3, 33, True, 40), (700, 4, 70, False, 150),
                                                       (900, 3, 130, True, 100)])
def test_every_shape_on_uneven_cells(n, cells, crowd, periodic, nb):
    s = _cloud(n, cells, crowd, periodic, nb)
    ref = None
    for v in range(max(N_BUILD_VARIANTS, N_FORCES_VARIANTS)):
        sim = sim_for(s, max_neibs=512)
        sim.set_variants(build=v % N_BUILD_VARIANTS, forces=v % N_FORCES_VARIANTS)
        sim.build_neighbors()
        counts, ids = sim.download_neighbors()
        sim.forces()
        got = (counts, ids, *sim.download_forces(), sim.stats()["list_entries"])
        if ref is None:
            ref = got
            compare_neighbor_sets(s, counts, ids)
        for a, b in zip(got, ref):
            assert np.array_equal(a, b, equal_nan=True) if isinstance(a, np.ndarray) else a == b
    # the default shapes of a state this small
    sim = sim_for(s, max_neibs=512)
    sim.forces()
    for a, b in zip(sim.download_forces(), ref[2:4]):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("max_neibs", [8, 33, 64, 65])
def test_every_build_cuts_a_full_list_at_the_same_entry(max_neibs):
    s = _cloud(600, 3, 90, True, 120, seed=2)
    ref = None
    for v in range(N_BUILD_VARIANTS):
        sim = sim_for(s, max_neibs=max_neibs)
        sim.set_variants(build=v)
        sim.build_neighbors()
        st = sim.stats(check=False)
        assert st["rc"] == -4
        got = (*sim.download_neighbors(), np.array([st["max_neibs_seen"], st["list_entries"]]))
        assert (got[0].sum(1) <= max_neibs).all()
        if ref is None:
            ref = got
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("visc", [0, 1])
@pytest.mark.parametrize("skin", [0.0, 0.3])
@pytest.mark.parametrize("walls", [False, True])
def test_density_diffusion_in_every_shape_matches_the_oracle(visc, skin, walls):
    # the default kernel, formulation and viscosities with density diffusion
    if walls:
        s = scenes.dam_break(dp=0.04)
        f = s.ptype == 0
        s.vel[f] = scenes.seeded_normal((int(f.sum()), 3), 0.05, 5).astype(np.float32)
    else:
        s = scenes.periodic_box(n_per_axis=12, jitter=0.2, seed=6)
        s.delta = np.random.default_rng(7).uniform(-1e-3, 1e-3, s.n).astype(np.float32)
    s = dataclasses.replace(s, visc=visc, nu=1e-3 if visc else 0.0, ddiff=1, ddiff_coef=0.1)
    kw = dict(rebuild_every=10, skin=skin * s.h, max_neibs=224) if skin else {}
    a_ref, d_ref, mag = oracle.rhs(oracle.params(s), s.pos, s.vel, s.delta, s.mass, s.ptype, with_mag=True)
    ref = None
    for v in range(N_FORCES_VARIANTS):
        sim = sim_for(s, **kw)
        sim.set_variants(forces=v)
        sim.forces()
        acc, drho = sim.download_forces()
        rel_check(acc, a_ref, 1e-5, "acceleration", mag[:, 0])
        rel_check(drho, d_ref, 1e-5, "density rate", mag[:, 1])
        sim.step(3)
        got = (acc, drho, *sim.download())
        assert sim.stats()["error_bits"] == 0
        if ref is None:
            ref = got
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("skin", [False, True])
def test_runs_of_steps_equal_single_steps(skin):
    """Calls of several steps replay graphs of several, from either buffer: the same bits as one step a call."""
    s = _cloud(700, 4, 20, True, 60)
    kw = dict(rebuild_every=4, skin=0.3 * s.h, max_neibs=512) if skin else dict(max_neibs=512)
    a, b = sim_for(s, **kw), sim_for(s, **kw)
    for run in (3, 5, 4, 9, 1, 22, 4):  # below, at and above a graph's steps, odd and even; the graph is made in between
        a.step(run)
        for _ in range(run):
            b.step(1)
        for x, y in zip(a.download(), b.download()):
            assert np.array_equal(x, y)
    sa, sb = a.stats(), b.stats()
    assert sa["steps"] == sb["steps"] == 48 and sa["time"] == sb["time"] and sa["builds"] == sb["builds"]
    assert sa["kernels_per_step"] == sb["kernels_per_step"]


@pytest.mark.parametrize("n_axis", [9, 137])
def test_fused_build_and_predictor_by_size(n_axis):
    """The fused kernel that large uploads choose (2.57 million particles), and the one asked for: the bits
    of the two kernels; a build variant set ends the choice."""
    s = scenes.periodic_box(n_per_axis=n_axis, dp=0.02)
    large = s.n > 2_500_000
    a, f = sim_for(s), sim_for(s)
    assert f.step_options()["fused_predict"] == large
    a.set_variants(build=1)
    assert not a.step_options()["fused_predict"]
    if not large:
        f.set_fused_predict(True)
    for sim in (a, f):
        sim.step(3)
    for x, y in zip(a.download(), f.download()):
        assert np.array_equal(x, y)
    sa, sf = a.stats(), f.stats()
    assert sa["list_entries"] == sf["list_entries"] and sa["dt"] == sf["dt"]


@pytest.mark.parametrize("max_neibs,rows", [(256, True), (257, False)])
def test_lists_too_long_for_shared_memory_take_the_thread_build(max_neibs, rows):
    """The default of a small state, and what tuning may choose, by list length."""
    s = scenes.periodic_box(n_per_axis=16)
    sim = sim_for(s, max_neibs=max_neibs)
    assert sim.variants()["build"].startswith("warp/row" if rows else "thread/particle")
    sim.autotune()
    assert rows or sim.variants()["build"].startswith("thread/particle")


def test_crowded_cells_in_the_row_build():
    """Cells of more than 64 particles, several tiles per block: the thread build's lists, in no more than
    2.5 times its time (1.4 measured; 4.6 when one warp of each block built them)."""
    s = dataclasses.replace(scenes.periodic_box(n_per_axis=43, jitter=0.1, seed=3), h=1.9 * 0.02)
    sim = sim_for(s, max_neibs=256)
    assert s.n / sim.stats()["n_cells"] > 59  # candidate slots are aligned to four: over 64 beside most cells
    got, ms = [], []
    for v in (0, 4):
        sim.set_variants(build=v)
        sim.step_profiled(2)
        ms.append(min(sim.step_profiled(4)["build"] for _ in range(5)))
        sim.upload(s)
        got.append((*sim.download_neighbors(), sim.stats()["list_entries"]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert ms[1] < 2.5 * ms[0]


def _row_build_tiles(s):
    """Tiles of 32 sorted particles by what the build by rows does with them (lists of up to 256 entries):
    (kept in shared memory, of those beside a cell of over 32 candidate slots, put off)."""
    nc = np.floor(np.array(s.size) / (s.kernel_radius * s.h)).astype(int)
    c = np.minimum((s.pos / (np.array(s.size) / nc)).astype(int), nc - 1)
    key = c[:, 0] + nc[0] * (c[:, 1] + nc[1] * c[:, 2])
    order = np.lexsort((np.arange(s.n), s.ptype, key))
    start = np.searchsorted(key[order], np.arange(nc.prod() + 1))
    end = np.stack([start[1:], start[:-1] + np.bincount(key[s.ptype == 0], minlength=nc.prod())], 1)  # of a fluid, a wall particle
    slots = end - (start[:-1] & ~3)[:, None]
    slots[end - start[:-1, None] == 0] = 0
    most = np.zeros(s.n, int)  # of the neighbour cells' slots, by sorted particle
    for d in np.ndindex(3, 3, 3):
        q = c[order] + np.array(d) - 1
        ok = np.ones(s.n, bool)
        for a in range(3):
            if (s.periodic >> a) & 1:
                q[:, a] %= nc[a]
            else:
                ok &= (q[:, a] >= 0) & (q[:, a] < nc[a])
        q = np.where(ok[:, None], q, 0)
        k = q[:, 0] + nc[0] * (q[:, 1] + nc[1] * q[:, 2])
        most = np.maximum(most, np.where(ok, slots[k, s.ptype[order]], 0))
    tile = np.array([most[i:i + 32].max() for i in range(0, s.n, 32)])
    return int((tile <= 64).sum()), int(((tile <= 64) & (tile > 32)).sum()), int((tile > 64).sum())


@pytest.mark.parametrize("n,cells,crowd,periodic,nb,max_neibs,put_off",
                         [(700, 5, 33, True, 120, 256, False), (900, 5, 50, False, 250, 255, False),
                          (1201, 6, 52, True, 400, 129, False), (1500, 6, 90, True, 300, 256, True),
                          (1100, 6, 70, False, 300, 255, True)])
def test_row_build_in_shared_memory(n, cells, crowd, periodic, nb, max_neibs, put_off):
    """Lists put together in shared memory, beside cells of 33 to 64 slots (a second hit mask), alone and
    with put-off tiles in the same launch: the oracle's sets, and every variant one list."""
    s = _cloud(n, cells, crowd, periodic, nb, seed=n)
    kept, two_masks, off = _row_build_tiles(s)
    assert kept > 0 and (off > 0 if put_off else two_masks > 0 and off == 0), (kept, two_masks, off)
    ref = None
    for v in range(N_BUILD_VARIANTS):
        sim = sim_for(s, max_neibs=max_neibs)
        sim.set_variants(build=v)
        sim.build_neighbors()
        got = (*sim.download_neighbors(), sim.stats()["list_entries"], sim.stats()["max_neibs_seen"])
        if ref is None:
            ref = got
            compare_neighbor_sets(s, *got[:2])
        for a, b in zip(got, ref):
            assert np.array_equal(a, b) if isinstance(a, np.ndarray) else a == b


@pytest.mark.parametrize("max_neibs", [8, 17, 32, 33, 64, 65])
def test_row_build_cuts_lists_in_shared_memory(max_neibs):
    """The same lists cut at their last entry, in tiles that are kept in shared memory, fluid and wall parts."""
    s = _cloud(900, 5, 50, True, 400, seed=8)
    kept, two_masks, off = _row_build_tiles(s)
    assert kept > 0 and two_masks > 0 and off == 0
    full, _ = (lambda sim: (sim.build_neighbors(), sim.download_neighbors())[1])(sim_for(s, max_neibs=256))
    ref = None
    for v in range(N_BUILD_VARIANTS):
        sim = sim_for(s, max_neibs=max_neibs)
        sim.set_variants(build=v)
        sim.build_neighbors()
        st = sim.stats(check=False)
        assert st["rc"] == -4
        got = (*sim.download_neighbors(), np.array([st["max_neibs_seen"], st["list_entries"]]))
        assert np.array_equal(got[0].sum(1), np.minimum(full.sum(1), max_neibs))
        if ref is None:
            ref = got
            cut = full.sum(1) > max_neibs
            assert (got[0][cut] > 0).all(1).any()  # both parts in a list that is cut
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n_axis,threads", [(20, 128), (33, 32), (34, 64), (41, 64), (42, 128)])
def test_shape_of_accelerations_alone(n_axis, threads):
    """sph_forces by particle count: 8 lanes, 16 and 8 entries a round, plain, on lines of its own; a shape that is
    set holds for it too."""
    import torch
    s = scenes.periodic_box(n_per_axis=n_axis)
    sim = sim_for(s)
    stream = torch.cuda.Stream()
    sim.forces()
    torch.cuda.synchronize()
    assert launches(lambda: sim.forces(stream=stream), stream) == [threads]
    sim.set_variants(forces=2)
    sim.forces()
    torch.cuda.synchronize()
    assert launches(lambda: sim.forces(stream=stream), stream) == [256]
