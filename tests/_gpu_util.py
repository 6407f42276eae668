"""Shared helpers of the GPU parity tests: run the CUDA path through the C-ABI and
rebuild, from its outputs, the oracle state in the same (cell) order."""
import ctypes

import numpy as np

import oracle


def gpu_hydro(d: dict, **params):
    """build -> density -> force on the GPU.  Returns (ctx, parts, out dict, iters)."""
    from paper_1508_00115_gb300 import binding
    n = int(d["x"].size)
    params.setdefault("flags", binding.SPH_FLAG_NGB_HASH)
    ctx = binding.Context(n, **params)
    parts = binding.Particles(d)
    ctx.build_cells(parts)
    it = ctx.density(parts)
    ctx.force(parts)
    out = parts.numpy()
    out["perm"] = ctx.permutation()
    out["iters"] = it
    if params["flags"] & binding.SPH_FLAG_NGB_HASH:
        out["ngb_hash"] = ctx.ngb_hash()
    out["stats"] = ctx.stats()
    return ctx, parts, out


def set_limit(ctx, which: int, value: int):
    """sph_test_limit: let something of the context run out early (-1: as it comes)."""
    from paper_1508_00115_gb300 import binding
    assert binding.lib().sph_test_limit(ctx.h, ctypes.c_int32(which), ctypes.c_int64(value)) == binding.SPH_OK


def force_pairs(parts) -> int:
    """Directed pairs r_ij < max(h_i, h_j), j != i, of the particles in a box of side 1 (FP64)."""
    import torch
    x = torch.stack([parts.t[c] for c in ("x", "y", "z")], dim=1)
    h, n, pairs = parts.t["h"].double(), x.shape[0], 0
    for i in range(0, n, 2000):
        dx = x[i:i + 2000, None] - x[None]
        r2 = ((dx - torch.round(dx)) ** 2).sum(dim=2)
        pairs += int((r2 < torch.maximum(h[i:i + 2000, None], h[None]) ** 2).sum())
    return pairs - n


def oracle_state(g: dict, box: float = 1.0) -> oracle.State:
    """FP64 oracle state from the GPU arrays (GPU order, GPU h, GPU ids)."""
    return oracle.State(x=g["x"], y=g["y"], z=g["z"], vx=g["vx"], vy=g["vy"], vz=g["vz"],
                        m=g["m"].astype(np.float64), u=g["u"].astype(np.float64),
                        h=g["h"].astype(np.float64), box=box,
                        ids=g["perm"].astype(np.uint64))


def rel(a, b):
    return np.abs(np.asarray(a, np.float64) - b) / np.abs(b)


def check_density(g, s, targets=None, rtol=1e-5, h_tol=1e-4):
    """Parity of the density pass at the GPU's smoothing lengths."""
    t = np.arange(s.n) if targets is None else np.asarray(targets)
    d = oracle.density_at_h(s, targets=t)
    assert rel(g["rho"][t], d["rho"]).max() <= rtol
    # h satisfies the criterion, rechecked in FP64 (FP32 rounding of h adds ~1e-6)
    assert np.abs(d["nw"] / 48.0 - 1).max() <= h_tol + 2e-6
    # neighbour sets: counts and set fingerprints exact
    assert np.array_equal(g["n_ngb"][t].astype(np.int64), d["n_ngb"])
    if "ngb_hash" in g:
        assert np.array_equal(g["ngb_hash"][t], d["ngb_hash"])
    # velocity estimates (feed only the viscosity switch): normalised by their RMS
    for k, gk in (("divv", g["divv"][t]), ("curl_abs", g["curl"][t])):
        scale = np.sqrt(np.mean(d[k] ** 2))
        if scale > 0:
            assert np.abs(gk - d[k]).max() <= 1e-4 * scale, k
    return d


def check_ghost(g, s, d, t, rtol=1e-5):
    gh = oracle.ghost(d["rho"], d["drho_dh"], d["divv"], d["curl_abs"], s.u[t], s.h[t])
    assert rel(g["P"][t], gh["P"]).max() <= rtol
    assert rel(g["c"][t], gh["c"]).max() <= 1e-6
    assert rel(g["f"][t], gh["f"]).max() <= 1e-4
    return gh


def check_force(g, s, targets=None, atol_rel=1e-4):
    """Force parity given the GPU density outputs (themselves checked above)."""
    t = np.arange(s.n) if targets is None else np.asarray(targets)
    # Balsara B from the GPU's divergence/curl (B needs neither f nor drho/dh);
    # P, c, f as the GPU computed them
    gh = oracle.ghost(g["rho"], np.zeros(s.n), g["divv"], g["curl"], s.u, s.h)
    fr = oracle.force(s, s.h, g["rho"].astype(np.float64), g["P"].astype(np.float64),
                      g["c"].astype(np.float64), g["f"].astype(np.float64), gh["B"],
                      targets=t)
    a = np.stack([g["ax"][t], g["ay"][t], g["az"][t]], axis=1).astype(np.float64)
    rms = np.sqrt(np.mean(np.sum(fr["a"] ** 2, axis=1)))
    err = np.sqrt(np.sum((a - fr["a"]) ** 2, axis=1)).max()
    assert err <= atol_rel * rms, (err, rms)
    du_rms = np.sqrt(np.mean(fr["dudt"] ** 2))
    if du_rms > 0:
        assert np.abs(g["dudt"][t] - fr["dudt"]).max() <= atol_rel * du_rms
    nz = fr["vsig"] > 0
    assert rel(g["vsig"][t][nz], fr["vsig"][nz]).max() <= 1e-5
    assert np.all(g["vsig"][t][~nz] == 0)
    return fr
