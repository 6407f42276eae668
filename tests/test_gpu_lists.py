"""Neighbour lists of the pair sums: one search serves the h iteration and the force
pass as long as no h leaves its list radius (4 % beyond the h of the search).  The cases
here start the second call from h that leave it: for a few particles (searched for one by
one, with the targets whose lists miss them) and for all of them (searched again as a
whole).  The bar is that of the other parity tests: neighbour sets exact."""
import numpy as np
import pytest

from paper_1508_00115_gb300 import inputs

from _gpu_util import check_density, check_force, force_pairs, oracle_state, set_limit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _second_call(d, flags, factor, share, **kw):
    """Converge, scale `share` of the h by `factor`, and run build, density and force again."""
    from paper_1508_00115_gb300 import binding
    n = int(d["x"].size)
    ctx = binding.Context(n, flags=flags | binding.SPH_FLAG_NGB_HASH, **kw)
    parts = binding.Particles(d)
    ctx.build_cells(parts)
    ctx.density(parts)
    ctx.force(parts)
    pick = torch.as_tensor(np.random.default_rng(5).random(n) < share, device="cuda")
    parts.t["h"][pick] *= factor
    ctx.build_cells(parts)
    ctx.density(parts)
    ctx.force(parts)
    g = parts.numpy()
    g["perm"], g["ngb_hash"], g["stats"] = ctx.permutation(), ctx.ngb_hash(), ctx.stats()
    return g


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("factor,share", [(0.9, 0.01), (0.9, 1.0), (1.2, 1.0), (0.6, 0.3)])
def test_h_leaving_its_list_radius(adaptive, factor, share):
    from paper_1508_00115_gb300 import binding
    if adaptive:
        d = inputs.plummer_mix(6000, seed=31, n_halos=6)
        flags = binding.SPH_FLAG_ADAPTIVE
    else:
        d = inputs.uniform(6000, seed=32)
        flags = 0
    d = inputs.random_velocities(d, 0.3, 33)
    g = _second_call(d, flags, factor, share, cell_factor=1.5)
    s = oracle_state(g)
    check_density(g, s)
    check_force(g, s)


def test_sums_do_not_depend_on_the_lists_beside_them():
    """Targets left for a second pass come in any order, four to a warp: every output has the
    same bits whichever lists share the warp."""
    from paper_1508_00115_gb300 import binding
    d = inputs.random_velocities(inputs.uniform(40000, seed=5), 0.3, 6)
    first = None
    for _ in range(12):
        g = _second_call(d, 0, 0.9, 0.02, cell_factor=1.25)
        g.pop("stats")
        first = first or g
        for k, v in g.items():
            assert np.array_equal(v, first[k]), k


@pytest.mark.parametrize("n", [200, 257, 1031])
@pytest.mark.parametrize("tw", [0, 16])
def test_lists_of_small_sets(n, tw):
    """Partial tiles and batches, the pages' edges, stencils that span the box."""
    from paper_1508_00115_gb300 import binding
    d = inputs.random_velocities(inputs.uniform(n, seed=n), 0.2, n + 1)
    g = _second_call(d, binding.SPH_FLAG_ADAPTIVE, 0.97, 1.0, tile_width=tw, leaf_max=32)
    s = oracle_state(g)
    check_density(g, s)
    check_force(g, s)


def test_lists_of_thousands_of_names():
    """A dense clump of 3,000 inside the kernel of sparse particles: lists beyond the eight
    lanes' share (the whole warp takes them) and over several chunks."""
    from paper_1508_00115_gb300 import binding
    rng = np.random.default_rng(9)
    d = inputs.random_velocities(inputs.uniform(4000, seed=41), 0.2, 42)
    for k in ("x", "y", "z"):
        d[k][:3000] = 0.5 + 0.002 * (rng.random(3000) - 0.5)
    g = _second_call(d, binding.SPH_FLAG_ADAPTIVE | binding.SPH_FLAG_TREE_H_GUESS, 0.98, 1.0)
    assert g["n_ngb"].max() > 1000
    s = oracle_state(g)
    check_density(g, s)
    check_force(g, s)


def test_leaf_too_large_for_its_names():
    """Groups of four coincident particles with leaves of at most two: a name holds the
    indices 0 and 1 only, and the sums run without lists."""
    from paper_1508_00115_gb300 import binding
    d = inputs.random_velocities(inputs.uniform(2000, seed=51), 0.2, 52)
    for k in ("x", "y", "z"):
        d[k][:12] = np.repeat(d[k][:3], 4)
    g = _second_call(d, binding.SPH_FLAG_ADAPTIVE, 1.0, 0.0, leaf_max=2)
    s = oracle_state(g)
    check_density(g, s)
    check_force(g, s)
    # captured steps: each search finds the leaf, the sums run without lists
    ctx = binding.Context(2000, flags=binding.SPH_FLAG_ADAPTIVE | binding.SPH_FLAG_NGB_HASH, leaf_max=2)
    parts = binding.Particles(d)
    for _ in range(3):
        ctx.steps(parts, 2, 1e-6)
        assert ctx.stats()["graph_steps"] > 0
        _check_call(ctx, parts)


def _lowered(parts, share, factor, seed):
    pick = torch.as_tensor(np.random.default_rng(seed).random(parts.t["h"].numel()) < share, device="cuda")
    parts.t["h"][pick] *= factor


@pytest.mark.parametrize("flag", ["uniform", "adaptive", "autotune"])
def test_density_calls_that_no_force_follows(flag):
    """The targets a density call marks for the force pass's search are that call's alone: calls
    without a force pass after them (and the tuner's own) leave nothing to the next."""
    from paper_1508_00115_gb300 import binding
    flags = {"uniform": 0, "adaptive": binding.SPH_FLAG_ADAPTIVE, "autotune": binding.SPH_FLAG_AUTOTUNE}[flag]
    d = inputs.plummer_mix(6000, seed=61, n_halos=6) if flag == "adaptive" else inputs.uniform(6000, seed=62)
    d = inputs.random_velocities(d, 0.3, 63)
    ctx = binding.Context(6000, flags=flags | binding.SPH_FLAG_NGB_HASH, cell_factor=1.5)
    parts = binding.Particles(d)
    for k in range(5):
        ctx.build_cells(parts)
        ctx.density(parts)
        _lowered(parts, 0.01, 0.9, 64 + k)
    ctx.build_cells(parts)
    ctx.density(parts)
    ctx.force(parts)
    g = parts.numpy()
    g["perm"], g["ngb_hash"] = ctx.permutation(), ctx.ngb_hash()
    s = oracle_state(g)
    check_density(g, s)
    check_force(g, s)


def test_source_that_grows_past_a_capped_list_radius():
    """Adaptive cells: a list ends at 1.15 of the leaf's largest h at the build, here below 1.04 of
    the (predicted) h that the search took for the source's reach.  Particles that grow from
    0.92 of theirs into that gap are missed by the neighbour's list, and its force sum has to get
    them: the pairs of the force pass against all pairs in FP64."""
    from paper_1508_00115_gb300 import binding
    n = 20000
    d = inputs.random_velocities(inputs.uniform(n, seed=71), 0.1, 72)
    at = np.linspace(0.0, 1.0, 4097)  # density exp(2 cos 2 pi x): h changes by a third within h
    mass = np.cumsum(np.exp(2.0 * np.cos(2.0 * np.pi * at)))
    d["x"] = np.interp(d["x"], (mass - mass[0]) / (mass[-1] - mass[0]), at)
    ctx = binding.Context(n, flags=binding.SPH_FLAG_ADAPTIVE | binding.SPH_FLAG_HPREDICT, cell_factor=1.25,
                          leaf_max=32, h_tol=1e-5)
    f = np.zeros(binding.SPH_HP_NF32, np.float32)
    f[135:141] = 1.0
    f[141] = np.log(1.149)  # every h is predicted to grow by that
    f[142] = 1.0
    ctx.hp_load(np.zeros(binding.SPH_HP_NBF16, np.uint16), f)
    parts = binding.Particles(d)
    kept = 0
    for k in range(8):
        ctx.build_cells(parts)
        ctx.density(parts)
        ctx.force(parts)
        _lowered(parts, 0.003, 0.8, 73 + k)
        ctx.reset_stats()
        ctx.step(parts, 1e-9)
        st = ctx.stats()
        kept += st["rebuilds"] == 0  # (a rebuild starts from the grown h)
        assert st["force_pairs"] == force_pairs(parts), k
    assert kept >= 3


def _call(ctx, parts, factor):
    """Build, density and force with every h scaled by factor; whether the sums ran over lists
    (without them a pass evaluates a target once)."""
    parts.t["h"] *= factor
    ctx.build_cells(parts)
    ctx.reset_stats()
    ctx.density(parts)
    st = ctx.stats()
    ctx.force(parts)
    return st["density_targets"] > parts.t["h"].numel() * st["density_passes"]


def _check_call(ctx, parts):
    g = parts.numpy()
    g["perm"], g["ngb_hash"] = ctx.permutation(), ctx.ngb_hash()
    s = oracle_state(g)
    check_density(g, s)
    check_force(g, s)


@pytest.mark.parametrize("adaptive", [False, True])
def test_pool_without_room_to_grow(adaptive):
    """No device memory for a larger pool: the call that needs one runs without lists, and the
    pool at hand serves those after it.  None for any pool: lists once there is."""
    from paper_1508_00115_gb300 import binding
    d = inputs.random_velocities(inputs.uniform(6000, seed=81), 0.3, 82)
    flags = binding.SPH_FLAG_NGB_HASH | (binding.SPH_FLAG_ADAPTIVE if adaptive else 0)
    ctx = binding.Context(6000, flags=flags)
    parts = binding.Particles(d)
    _call(ctx, parts, 1.0)
    assert _call(ctx, parts, 0.98)
    set_limit(ctx, 1, 0)
    assert not _call(ctx, parts, 2.0)  # lists of 430 names: 14 pages, and the pool has 5 per particle
    _check_call(ctx, parts)
    assert _call(ctx, parts, 0.98)
    _check_call(ctx, parts)
    ctx = binding.Context(6000, flags=flags)
    set_limit(ctx, 1, 0)
    parts = binding.Particles(d)
    _call(ctx, parts, 1.0)
    assert not _call(ctx, parts, 0.98)
    _check_call(ctx, parts)
    ctx.steps(parts, 2, 1e-6)
    set_limit(ctx, 1, -1)
    _call(ctx, parts, 0.98)
    assert _call(ctx, parts, 0.98)
    ctx.steps(parts, 2, 1e-6)
    ctx.build_cells(parts)
    ctx.density(parts)
    ctx.force(parts)
    _check_call(ctx, parts)


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("pages", [1.0, 2.0, 2.5, 3.0, 3.5, 4.0, 5.0])
def test_pool_that_runs_out(adaptive, pages):
    """Pools of too few pages per particle: they run out in the first search, in that of the
    targets whose h left its list, in that of a grown neighbour's, or not, outside captures and
    inside them; the sums are the same."""
    from paper_1508_00115_gb300 import binding
    n = 3000
    d = inputs.random_velocities(inputs.uniform(n, seed=91), 0.3, 92)
    flags = binding.SPH_FLAG_NGB_HASH | (binding.SPH_FLAG_ADAPTIVE if adaptive else 0)
    ctx = binding.Context(n, flags=flags, cell_factor=1.25)
    set_limit(ctx, 2, int(pages * n))
    parts = binding.Particles(d)
    for k, share in enumerate((0.0, 1.0, 0.03, 0.3, 0.03)):
        _lowered(parts, share, 0.9, 93 + k)
        ctx.build_cells(parts)
        ctx.density(parts)
        ctx.force(parts)
        _check_call(ctx, parts)
    for k in range(3):
        ctx.steps(parts, 2, 1e-4)
        ctx.build_cells(parts)
        ctx.density(parts)
        ctx.force(parts)
        _check_call(ctx, parts)


def test_lists_that_never_fit():
    """Lists that do not fit the largest pool: the search that shows it runs in ever fewer of
    the calls, and captured steps are captured again without it."""
    from paper_1508_00115_gb300 import binding
    n = 3000
    d = inputs.random_velocities(inputs.uniform(n, seed=95), 0.3, 96)
    ctx = binding.Context(n)
    set_limit(ctx, 2, n)
    parts = binding.Particles(d)
    launches = []
    for _ in range(17):
        parts.t["h"] *= 0.98
        ctx.build_cells(parts)
        ctx.reset_stats()
        ctx.density(parts)
        launches.append(ctx.stats()["kernel_launches"])
    tried = [v > min(launches) for v in launches]
    assert [k for k, t in enumerate(tried) if t] == [0, 1, 3, 6, 11], launches
    ctx = binding.Context(n)
    set_limit(ctx, 2, n)
    parts = binding.Particles(d)
    steps = []
    for _ in range(4):
        ctx.reset_stats()
        ctx.steps(parts, 3, 1e-6)
        steps.append(ctx.stats()["kernel_launches"])
    assert steps[1] == steps[3] < steps[2], steps  # (the first call's hydro pass has missed once)


@pytest.mark.parametrize("n,factor", [(1200, 1.3), (4000, 1.35), (4000, 1.5), (4000, 2.0), (6000, 2.4)])
def test_guesses_above_the_root(n, factor):
    """First calls whose guess asks for more names than the pool holds: passes without lists
    until the lists will be short, then one search for all."""
    from paper_1508_00115_gb300 import binding
    d = inputs.random_velocities(inputs.uniform(n, seed=101), 0.3, 102)
    ctx = binding.Context(n, flags=binding.SPH_FLAG_NGB_HASH)
    parts = binding.Particles(d)
    _call(ctx, parts, factor)
    _check_call(ctx, parts)
    assert _call(ctx, parts, 0.97)
    _check_call(ctx, parts)


@pytest.mark.parametrize("factor", [0.7, 0.9, 0.99, 1.1])
def test_iterations_are_evaluations(factor):
    """sph_density reports the evaluations of the h iteration, as many with lists, which iterate
    within a pass, as without (no room for them): one may differ where a target ends at h_tol."""
    from paper_1508_00115_gb300 import binding
    d = inputs.uniform(6000, seed=111)
    its = []
    for free in (-1, 0):
        ctx = binding.Context(6000, cell_factor=1.5)
        set_limit(ctx, 1, free)
        parts = binding.Particles(d)
        ctx.build_cells(parts)
        ctx.density(parts)
        parts.t["h"] *= factor
        ctx.build_cells(parts)
        its.append(ctx.density(parts))
    assert its[1] >= 2 and abs(its[0] - its[1]) <= 1, its


def test_pairs_closer_than_normal_squares():
    """Two particles 3e-20 apart (at a cell centre of a box of side 1e-3), whose squared distance
    is a denormal FP32 number, approach each other: the pair has its direction, and its signal
    velocity counts."""
    from paper_1508_00115_gb300 import binding
    n, box = 4000, 1e-3
    d = inputs.random_velocities(inputs.uniform(n, seed=121, box=box), 0.1, 122)
    nc = None
    for _ in range(2):
        ctx = binding.Context(n, box_size=box, flags=binding.SPH_FLAG_NGB_HASH)
        parts = binding.Particles(d)
        ctx.build_cells(parts)
        ctx.density(parts)
        ctx.force(parts)
        st, g = ctx.stats(), parts.numpy()
        g["perm"], g["ngb_hash"] = ctx.permutation(), ctx.ngb_hash()
        if nc is None:
            nc = st["nc"]
            c = 0.5 * (box / nc)
            for k in "xyz":
                d[k][:2] = c
            d["x"][1] = c + 2 * np.spacing(c)
            d["vx"][:2] = (5.0, -5.0)
    assert st["nc"] == nc and 0 < (d["x"][1] - d["x"][0]) ** 2 < 1.1e-38
    s = oracle_state(g, box)
    check_density(g, s)
    check_force(g, s)
    assert (g["vsig"][g["perm"] < 2] > 30).all()
