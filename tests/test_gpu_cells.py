"""The cell build's sort and prefix sums at the edges of their tiles: permutation and keys
equal a stable argsort of the keys of the input order, exactly."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1508_00115_gb300 import binding, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h", [(1, 0.2), (33, 0.3), (1023, 0.1), (1025, 0.05), (16385, 0.03), (131072, 0.02),
                                 (131073, 0.02), (262145, 0.012), (524288, 0.3), (524289, 0.008)])
def test_build_is_a_stable_sort_by_cell_and_octant(n, h):
    d = inputs.uniform(n, seed=n)
    d["h"] = np.full(n, h)
    ctx = binding.Context(n)
    parts = binding.Particles(d)
    ctx.build_cells(parts)
    nc = ctx.stats()["nc"]
    pos = [oracle.wrap(d[k], 1.0) for k in ("x", "y", "z")]
    cell = oracle.cell_keys(*pos, 1.0, nc).astype(np.int64)
    idx = (cell % nc, (cell // nc) % nc, cell // (nc * nc))
    octant = sum((p >= (i + 0.5) / nc).astype(np.int64) << b for b, (p, i) in enumerate(zip(pos, idx)))
    perm = np.argsort(cell * 8 + octant, kind="stable")
    assert np.array_equal(ctx.permutation(), perm)
    assert np.array_equal(ctx.cell_keys(), cell[perm])
    ctx.close()


@pytest.mark.parametrize("n", [900, 20000])
def test_adaptive_build_keeps_every_particle(n):
    d = inputs.plummer_mix(n, seed=n, n_halos=3)
    ctx = binding.Context(n, flags=binding.SPH_FLAG_ADAPTIVE)
    parts = binding.Particles(d)
    ctx.build_cells(parts)
    perm = ctx.permutation()
    assert np.array_equal(np.sort(perm), np.arange(n))
    assert np.array_equal(parts.numpy()["x"], d["x"][perm])
    ctx.close()


@pytest.mark.parametrize("n,leaf", [(900, 2), (3000, 8), (5000, 300), (120000, 8)])
def test_device_sized_trees_step_like_host_built_ones(n, leaf):
    """Captured steps build the tree a level per launch with its sizes on the device (beyond
    65,536 possible frontier nodes in several), host steps with host reads: deep trees, trees
    of roots only, joined octants.  Tolerances: test_gpu_adaptive.py."""
    from test_gpu_adaptive import _RT_RHO, _RT_STEPS, _same_state
    d = inputs.uniform(n, seed=n) if n < 1000 else inputs.plummer_mix(n, seed=n, n_halos=4)
    d = inputs.random_velocities(d, 0.2, 3)
    out = []
    for captured in (False, True):
        ctx = binding.Context(n, flags=binding.SPH_FLAG_ADAPTIVE, h_tol=1e-6, leaf_max=leaf, max_h_iter=60)
        parts = binding.Particles(d)
        if captured:
            ctx.steps(parts, 2, 1e-7)
            assert ctx.stats()["graph_steps"] == 2
        else:
            ctx.step(parts, 1e-7)
            ctx.step(parts, 1e-7)
        out.append((parts.numpy(), ctx.permutation()))
        ctx.close()
    _same_state(out[0][0], out[1][0], out[0][1], out[1][1], _RT_STEPS, _RT_RHO)


@pytest.mark.parametrize("adaptive", [False, True])
def test_captured_steps_after_the_scratch_was_replaced(adaptive):
    """A context that grows to more particles and comes back replays nothing that it captured with
    the arrays it had before."""
    n = 1500
    d = inputs.random_velocities(inputs.uniform(n, seed=7), 0.2, 8)
    out = []
    for grow in (False, True):
        ctx = binding.Context(n, flags=binding.SPH_FLAG_ADAPTIVE if adaptive else 0)
        parts = binding.Particles(d)
        ctx.steps(parts, 2, 1e-5)
        if grow:
            for m in (4 * n, n):
                assert binding.lib().sph_set_n(ctx.h, ctypes.c_int64(m)) == binding.SPH_OK
        else:
            ctx.build_cells(parts)  # (as a new particle count does, the next call starts with a hydro pass)
        ctx.steps(parts, 2, 1e-5)
        out.append(parts.numpy())
        ctx.close()
    for k in ("x", "vx", "u", "h", "rho", "ax"):
        assert np.array_equal(np.sort(out[0][k]), np.sort(out[1][k])), k
