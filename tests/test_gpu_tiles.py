"""The tiled force kernels (tensor-core pair filter) against the row walk.

DCM_FORCE_AUTO runs over tiles of 32 particles where they serve (boxes of at
least 4 rc_max, more than 32,768 particles in the mixed form); DCM_FORCE_PACKED
and DCM_FORCE_THREAD run the row walk.  Both accept the same pairs and evaluate each
with the same roundings, and differ in the order of the sums only.

Tolerances, from the order of the sums: a particle's force is a sum of partial
sums of at most about 40 FP32 terms (each within 40 x 2^-24 = 2.4e-6 of its
terms' magnitude, random signs: about 2^-24 sqrt(40) = 4e-7), the partial sums
added with compensation: RMS 1e-6 of the RMS force (mixed); FP64: 40 x 2^-53
rounded up, 1e-13.  Pair counts agree exactly.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MIXED_RMS, FP64_RMS = 1e-6, 1e-13


@pytest.fixture(scope="module")
def D():
    import paper_1701_05242_gb300.dcm as dcm
    return dcm


def lattice(box, seed, spacing=1.12, jitter=0.2):
    """Jittered simple cubic sites in the middle half of the box along z, a
    few far apart elsewhere: at least spacing - 2 jitter apart."""
    rng = np.random.default_rng(seed)
    n = [max(1, int(L / spacing)) for L in box]
    g = np.stack(np.meshgrid(*[(np.arange(k) + 0.5) * (L / k) for k, L in zip(n, box)], indexing="ij"), -1)
    g = g.reshape(-1, 3) + rng.uniform(-jitter, jitter, (np.prod(n), 3))
    dense = np.abs(g[:, 2] - 0.5 * box[2]) < 0.25 * box[2]
    g = g[dense | (rng.random(len(g)) < 0.03)]
    p = np.mod(g, np.array(box)).astype(np.float32)
    return np.minimum(p, np.nextafter(np.array(box, np.float32), np.float32(0)))


def cutoffs(pos, box, kind, rng):
    if kind == "ramp":
        depth = 0.25 * box[2] - np.abs(pos[:, 2] - 0.5 * box[2])
        return np.clip(6.0 - depth, 3.0, 6.0)
    if kind == "uniform":
        return np.full(len(pos), 3.0)
    return rng.choice([0.0, 2.5, 3.0, 4.7, 6.0], len(pos))  # mixed within every tile


def forces(D, box, pos, rc, types=None, prec="mixed", **kw):
    real = torch.float32 if prec == "mixed" else torch.float64
    n = len(pos)
    p = D.make_params(box, n_max=n, precision=D.DCM_PREC_MIXED if prec == "mixed" else D.DCM_PREC_FP64, **kw)
    ctx = D.Context(p)
    pos4 = D.to_real4(torch.from_numpy(pos), None if types is None else torch.from_numpy(types), real)
    dev = dict(dtype=torch.int32, device="cuda")
    cell, start, perm = torch.empty(n, **dev), torch.empty(ctx.ncell + 1, **dev), torch.empty(n, **dev)
    ps = torch.empty_like(pos4)
    D.dcm_bin(ctx, n, pos4, cell, start, perm, ps)
    rcs = torch.from_numpy(rc).to(real).cuda()[perm.long()].contiguous()
    F = torch.full_like(ps, 7.0)
    tot = torch.zeros(3, dtype=torch.float64, device="cuda")
    D.dcm_forces(ctx, n, ps, rcs, start, F, tot)
    torch.cuda.synchronize()
    assert D.dcm_status(ctx) == D.DCM_OK
    ctx.close()
    return F.double().cpu().numpy(), tot.cpu().numpy()


CASES = [
    # box, cell edges, cutoffs, two types, shift: bundles with a last single
    # row, rows of one cell step, several cells per rc, cells as wide as rc
    ((48.0, 45.0, 51.0), dict(), "ramp", False, 0),
    ((25.5, 64.5, 70.5), dict(lx=0.5), "ramp", False, 1),
    ((24.0, 61.5, 75.0), dict(lx=0.75), "mixed", True, 1),
    ((48.0, 46.5, 49.5), dict(l=0.75), "ramp", True, 0),
    ((48.0, 51.0, 45.0), dict(l=3.0, h=1.5), "uniform", False, 1),
    ((192.0, 24.0, 25.5), dict(lx=0.5), "mixed", False, 0),
]


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("box,edges,kind,typed,shift", CASES)
def test_tiles_equal_the_row_walk(D, box, edges, kind, typed, shift, prec):
    pos = lattice(box, 3)
    rng = np.random.default_rng(4)
    rc = cutoffs(pos, box, kind, rng)
    assert len(pos) > 32768
    kw = dict(edges, shift_energy=shift)
    types = None
    if typed:
        types = rng.integers(0, 2, len(pos)).astype(np.float32)
        kw.update(ntypes=2, eps=(1.0, 0.8), sigma=(1.0, 1.1))
    walk = D.DCM_FORCE_PACKED if prec == "mixed" else D.DCM_FORCE_THREAD
    F0, t0 = forces(D, box, pos, rc, types, prec, force_kernel=walk, **kw)
    F1, t1 = forces(D, box, pos, rc, types, prec, **kw)
    assert t1[2] == t0[2]
    tol = MIXED_RMS if prec == "mixed" else FP64_RMS
    rms = np.sqrt((F0[:, :3] ** 2).mean())
    assert np.sqrt(((F1 - F0)[:, :3] ** 2).mean()) <= tol * rms
    assert np.sqrt(((F1 - F0)[:, 3] ** 2).mean()) <= tol * np.sqrt((F0[:, 3] ** 2).mean()) * 4
    # totals: the particles' errors add up like sqrt(n)
    scale = np.abs(F0[:, 3]).sum()
    assert abs(t1[0] - t0[0]) <= 4 * tol * scale


def test_tiles_crowded_cells_and_empty_regions(D):
    """One cell with hundreds of particles (several full tiles from one cell
    step), everything else a thin gas: tiles end at their longest, lists
    overflow their chunk many times."""
    box = (96.0, 60.0, 60.0)
    rng = np.random.default_rng(8)
    g = np.stack(np.meshgrid(*[np.arange(9)] * 3, indexing="ij"), -1).reshape(-1, 3)
    clump = np.array([30.1, 15.1, 12.1]) + 0.15 * g + rng.uniform(-0.03, 0.03, (len(g), 3))
    gas = lattice(box, 9, spacing=2.1, jitter=0.5)
    gas = gas[np.abs(gas - np.array([30.7, 15.7, 12.7])).max(1) > 1.5]
    fill = lattice(box, 10, spacing=1.9, jitter=0.3)
    fill = fill[np.abs(fill - np.array([30.7, 15.7, 12.7])).max(1) > 2.5]
    pos = np.concatenate([clump, gas, fill]).astype(np.float32)
    pos = pos[rng.permutation(len(pos))]
    rc = rng.choice([3.0, 6.0], len(pos))
    assert len(pos) > 32768
    F0, t0 = forces(D, box, pos, rc, force_kernel=D.DCM_FORCE_PACKED, lx=0.5)
    F1, t1 = forces(D, box, pos, rc, lx=0.5)
    assert t1[2] == t0[2]
    scale = np.sqrt((F0[:, :3] ** 2).sum(1)).max()  # overlapping particles: one pair may outweigh all others
    assert np.abs(F1 - F0)[:, :3].max() <= 1e-6 * scale


@pytest.mark.parametrize("bad", [np.nan, np.inf, -3.0, 50.0, 1e30])
def test_tiles_coordinates_outside_the_box(D, bad):
    """A coordinate that is not in the box sends its own tile and every tile
    that meets it to the row walk: same NaN set, same values elsewhere."""
    box = (48.0, 45.0, 48.0)
    pos = lattice(box, 5)
    rng = np.random.default_rng(6)
    for k in rng.choice(len(pos), 7, replace=False):
        pos[k, rng.integers(0, 3)] = bad
    rc = np.full(len(pos), 3.0)
    F0, t0 = forces(D, box, pos, rc, force_kernel=D.DCM_FORCE_PACKED)
    F1, t1 = forces(D, box, pos, rc)
    assert np.array_equal(np.isnan(F0), np.isnan(F1))
    ok = ~np.isnan(F0).any(1)
    assert ok.sum() > 1000
    rms = np.sqrt((F0[ok, :3] ** 2).mean())
    assert np.sqrt(((F1 - F0)[ok, :3] ** 2).mean()) <= MIXED_RMS * rms
    if np.isfinite(t0).all():
        assert t1[2] == t0[2]
