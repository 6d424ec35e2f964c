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


def by_input(D, box, pos, rc, types, upstream=None, **kw):
    """Forces (or, with upstream gradients, the adjoint) in input order."""
    n = len(pos)
    fp64 = kw.get("precision") == D.DCM_PREC_FP64
    real = torch.float64 if fp64 else torch.float32
    ctx = D.Context(D.make_params(box, n_max=n, ntypes=2, eps=(1.0, 0.8), sigma=(1.0, 1.1), **kw))
    p4 = D.to_real4(torch.from_numpy(pos), torch.from_numpy(types), real)
    dev = dict(dtype=torch.int32, device="cuda")
    cell, start, perm = torch.empty(n, **dev), torch.empty(ctx.ncell + 1, **dev), torch.empty(n, **dev)
    ps = torch.empty_like(p4)
    D.dcm_bin(ctx, n, p4, cell, start, perm, ps)
    perm = perm.long()
    rcs = torch.from_numpy(rc).to(real).cuda()[perm].contiguous()
    out = torch.empty_like(ps)
    dpar = torch.zeros(4, dtype=torch.float64, device="cuda")
    if upstream is None:
        D.dcm_forces(ctx, n, ps, rcs, start, out)
    else:
        A = torch.from_numpy(upstream).to(real).cuda()[perm].contiguous()
        D.dcm_forces_backward(ctx, n, ps, rcs, start, A, 0.7, out, dpar)
    res = torch.empty_like(out)
    res[perm] = out
    assert D.dcm_status(ctx) == D.DCM_OK
    ctx.close()
    return res.double().cpu().numpy(), dpar.cpu().numpy()


def crossing(n_small, seed):
    """n_small particles, and the same with one more, alone in the vapor
    beyond everybody's cutoff."""
    box = (63.0, 61.5, 72.0)
    pos = lattice(box, seed)
    pos = pos[np.abs(pos[:, 2] - 36.0) < 18.0]
    rng = np.random.default_rng(seed)
    pos = pos[rng.permutation(len(pos))]
    assert len(pos) > n_small
    pos = pos[:n_small]
    rc = np.clip(6.0 - (18.0 - np.abs(pos[:, 2] - 36.0)), 3.0, 6.0)
    types = rng.integers(0, 2, n_small + 1).astype(np.float32)
    lone = np.array([[30.0, 30.0, 1.0]], np.float32)
    return box, np.concatenate([pos, lone]), np.append(rc, 6.0), types, rng


@pytest.mark.parametrize("lx", [0.0, 0.5])
def test_forces_on_both_sides_of_the_switch_to_tiles(D, lx):
    """32,768 particles run 16 lanes per particle, one more runs tiles."""
    n = 32768
    box, pos, rc, types, _ = crossing(n, 21)
    F0, _ = by_input(D, box, pos[:n], rc[:n], types[:n], lx=lx)
    F1, _ = by_input(D, box, pos, rc, types, lx=lx)
    assert np.all(F1[n] == 0.0)
    rms = np.sqrt((F0[:, :3] ** 2).mean())
    assert np.sqrt(((F1[:n] - F0)[:, :3] ** 2).mean()) <= MIXED_RMS * rms


@pytest.mark.parametrize("n,lx", [(3000, 0.0), (49152, 0.5), (49153, 0.5), (49153, 0.0)])
def test_adjoint_forms_against_fp64(D, n, lx):
    """A warp per particle (up to 49,152) and tiles (above) against the FP64
    row walk.  A pair term g'/r d d.A carries about 20 roundings, amplified by the
    powers of 1/r^2 (14 at most): 20 x 14 x 2^-24 = 1.7e-5 at worst, random over
    the pairs: RMS 5e-6; parameter sums over all pairs likewise."""
    box, pos, rc, types, rng = crossing(n - 1, 31)
    A = np.concatenate([rng.normal(size=(n, 3)), np.zeros((n, 1))], 1).astype(np.float32)
    # pairs whose distance is within FP32 rounding of a cutoff may fall on either side: their terms are of the
    # size of the forces at the cutoff, 1e-3 of the RMS gradient, and rare
    G0, d0 = by_input(D, box, pos, rc.astype(np.float32).astype(np.float64), types, A, lx=lx, shift_energy=1,
                      precision=D.DCM_PREC_FP64)
    G1, d1 = by_input(D, box, pos, rc.astype(np.float32).astype(np.float64), types, A, lx=lx, shift_energy=1)
    rms = np.sqrt((G0[:, :3] ** 2).mean())
    assert np.sqrt(((G1 - G0)[:, :3] ** 2).mean()) <= 5e-6 * rms
    assert np.all(G1[:, 3] == 0.0)
    assert np.all(np.abs(d1 - d0) <= 5e-6 * np.abs(d0).max())


@pytest.mark.parametrize("box,n,spacing,typed,kw", [
    ((42.0, 45.0, 51.0), None, 1.12, False, dict(lx=0.5)),              # tiles across every boundary
    ((33.0, 34.5, 40.5), None, 1.12, True, dict()),                     # most tiles at a boundary, two types
    ((42.0, 45.0, 51.0), None, 1.12, False, dict(newton3=1)),           # half lists
    ((33.0, 34.5, 40.5), None, 1.12, True, dict(newton3=1, lx=0.75)),
    ((33.0, 34.5, 40.5), None, 0.8, False, dict(lx=0.5)),               # denser than the capacity bound: two fills
    ((42.0, 45.0, 51.0), 4000, 1.12, False, dict(shift_energy=1)),      # the switch to tiles
    ((42.0, 45.0, 51.0), 3999, 1.12, False, dict(shift_energy=1)),
])
def test_lists_over_tiles(D, box, n, spacing, typed, kw):
    """Neighbour lists built over tiles against the cell path: the same pairs
    exactly; forces to 1e-5 (sums of up to 500 FP32 terms in one chain: 2^-24
    sqrt(500) = 1.3e-6 of partial sums a few times the force)."""
    pos = lattice(box, 41, spacing, 0.2 * spacing / 1.12)
    rng = np.random.default_rng(41)
    if n:
        pos = pos[rng.permutation(len(pos))[:n]]
    types = rng.integers(0, 2, len(pos)).astype(np.float32) if typed else None
    if typed:
        kw = dict(kw, ntypes=2, eps=(1.0, 0.8), sigma=(1.0, 1.1))
    res = []
    for skin in (0.5, 0.0):
        k = dict(kw) if skin else {a: b for a, b in kw.items() if a != "newton3"}
        ctx = D.Context(D.make_params(box, n_max=len(pos), recompute_every=4, skin=skin, **k))
        st = D.State(ctx, D.to_real4(torch.from_numpy(pos), None if types is None else torch.from_numpy(types)),
                     torch.zeros(len(pos), 4))
        D.dcm_step_init(ctx, st)
        for _ in range(2):  # a step so short that nothing moves
            D.dcm_step(ctx, st, 1e-12, 1)
        assert D.dcm_status(ctx) == D.DCM_OK
        _, _, rc, ids = st.current()
        F, r = np.empty((len(pos), 3)), np.empty(len(pos))
        ids = ids.cpu().numpy()
        F[ids], r[ids] = st.force.double().cpu().numpy()[:, :3], rc.double().cpu().numpy()
        res.append((F, r, st.thermo.cpu().numpy()))
        ctx.close()
    (F0, r0, t0), (F1, r1, t1) = res
    assert np.array_equal(r0, r1)
    assert t0[3] == t1[3]
    assert np.sqrt(((F0 - F1) ** 2).mean()) <= 1e-5 * np.sqrt((F1 ** 2).mean())
    assert abs(t0[0] - t1[0]) <= 1e-5 * abs(t1[0]) and abs(t0[1] - t1[1]) <= 1e-5 * abs(t1[1])


def with_negative_zeros(box, seed):
    """The lattice with some coordinates of -0.0 per axis (particles next to
    the boundary moved onto it, and those alone: nobody else within 0.9)."""
    pos = lattice(box, seed)
    rng = np.random.default_rng(seed)
    L = np.array(box, np.float32)
    keep = np.ones(len(pos), bool)
    on = []
    for d in range(3):
        near = np.flatnonzero(keep & (pos[:, d] < 0.9))
        for k in rng.choice(near, min(40, len(near)), replace=False):
            if keep[k]:
                pos[k, d] = -0.0
                dist = np.abs(pos - pos[k])
                dist = np.minimum(dist, L - dist)
                close = (dist ** 2).sum(1) < 0.81
                close[k] = False
                keep &= ~close
                on.append((k, d))
    on = [(k, d) for k, d in on if keep[k]]
    for d in range(3):
        assert sum(e == d for _, e in on) >= 10
    pos = pos[keep]
    assert (np.signbit(pos) & (pos == 0)).sum() >= 30
    return pos


@pytest.mark.parametrize("form", ["mixed", "fp64", "adjoint", "lists"])
@pytest.mark.parametrize("lx", [0.0, 0.5])
def test_coordinates_of_negative_zero(D, form, lx):
    """-0.0 lies in [0, L): the tiles that hold it reach as far as with +0.0."""
    box = (48.0, 60.0, 72.0)
    pos = with_negative_zeros(box, 71)
    rng = np.random.default_rng(72)
    rc = cutoffs(pos, box, "ramp", rng)
    assert len(pos) > 49152
    if form in ("mixed", "fp64"):
        walk = D.DCM_FORCE_PACKED if form == "mixed" else D.DCM_FORCE_THREAD
        F0, t0 = forces(D, box, pos, rc, prec=form, force_kernel=walk, lx=lx)
        F1, t1 = forces(D, box, pos, rc, prec=form, lx=lx)
        assert t1[2] == t0[2]
        tol = MIXED_RMS if form == "mixed" else FP64_RMS
        assert np.sqrt(((F1 - F0)[:, :3] ** 2).mean()) <= tol * np.sqrt((F0[:, :3] ** 2).mean())
    elif form == "adjoint":  # bounds as in test_adjoint_forms_against_fp64
        types = rng.integers(0, 2, len(pos)).astype(np.float32)
        A = np.concatenate([rng.normal(size=(len(pos), 3)), np.zeros((len(pos), 1))], 1).astype(np.float32)
        rc = rc.astype(np.float32).astype(np.float64)
        G0, d0 = by_input(D, box, pos, rc, types, A, lx=lx, precision=D.DCM_PREC_FP64)
        G1, d1 = by_input(D, box, pos, rc, types, A, lx=lx)
        assert np.sqrt(((G1 - G0)[:, :3] ** 2).mean()) <= 5e-6 * np.sqrt((G0[:, :3] ** 2).mean())
        assert np.all(np.abs(d1 - d0) <= 5e-6 * np.abs(d0).max())
    else:
        res = []
        for skin in (0.5, 0.0):
            ctx = D.Context(D.make_params(box, n_max=len(pos), skin=skin, lx=lx))
            st = D.State(ctx, D.to_real4(torch.from_numpy(pos)), torch.zeros(len(pos), 4))
            D.dcm_step_init(ctx, st)
            assert D.dcm_status(ctx) == D.DCM_OK
            ids = st.current()[3].cpu().numpy()
            F = np.empty((len(pos), 3))
            F[ids] = st.force.double().cpu().numpy()[:, :3]
            res.append((F, st.thermo.cpu().numpy()))
            ctx.close()
        (F0, t0), (F1, t1) = res
        assert t0[3] == t1[3]
        assert np.sqrt(((F0 - F1) ** 2).mean()) <= 1e-5 * np.sqrt((F1 ** 2).mean())


@pytest.mark.parametrize("prec,typed", [("mixed", False), ("mixed", True), ("fp64", False), ("fp64", True)])
@pytest.mark.parametrize("box,outside", [
    ((61.5, 25.5, 70.5), 0),    # tiles that reach past both ends of y
    ((70.5, 61.5, 25.5), 0),    # of z
    ((25.5, 25.5, 150.0), 0),   # of x and y
    ((48.0, 45.0, 51.0), 1),    # one bundle with a coordinate outside the box
    ((48.0, 45.0, 51.0), 60),   # most tiles next to one
])
def test_tiles_left_to_the_row_walk(D, box, outside, prec, typed):
    """Tiles that the filter does not serve, a few or most of them."""
    pos = lattice(box, 51)
    rng = np.random.default_rng(52)
    for k in rng.choice(len(pos), outside, replace=False):
        d = rng.integers(0, 3)
        pos[k, d] = rng.choice([-0.25, box[d], box[d] + 0.75])
    rc = cutoffs(pos, box, "mixed" if typed else "ramp", rng)
    assert len(pos) > 32768
    kw, types = dict(shift_energy=1), None
    if typed:
        types = rng.integers(0, 2, len(pos)).astype(np.float32)
        kw.update(ntypes=2, eps=(1.0, 0.8), sigma=(1.0, 1.1))
    walk = D.DCM_FORCE_PACKED if prec == "mixed" else D.DCM_FORCE_THREAD
    F0, t0 = forces(D, box, pos, rc, types, prec, force_kernel=walk, **kw)
    F1, t1 = forces(D, box, pos, rc, types, prec, **kw)
    assert t1[2] == t0[2]
    tol = MIXED_RMS if prec == "mixed" else FP64_RMS
    # one particle on top of another may outweigh all others: particle by particle, against the larger of its own
    # force and the RMS without the largest
    mag = np.sqrt((F0[:, :3] ** 2).sum(1))
    rms = np.sqrt((np.sort(mag)[:-200] ** 2).mean())
    err = np.sqrt(((F1 - F0)[:, :3] ** 2).sum(1)) / np.maximum(mag, rms)
    assert np.sqrt((err ** 2).mean()) <= tol and err.max() <= 40 * tol
    assert abs(t1[0] - t0[0]) <= 4 * tol * np.abs(F0[:, 3]).sum()


@pytest.mark.parametrize("ntypes", [1, 2])
@pytest.mark.parametrize("box,outside", [
    ((63.0, 61.5, 72.0), 0),    # hardly any tile left over
    ((64.5, 25.5, 102.0), 0),   # tiles that reach past both ends of y
    ((63.0, 61.5, 72.0), 1),
    ((63.0, 61.5, 72.0), 60),
])
def test_adjoint_tiles_left_to_the_row_walk(D, box, outside, ntypes):
    """The tiled adjoint and the kernel for the tiles left over, whose
    parameter sums share one table, against the FP64 row walk: bounds as in
    test_adjoint_forms_against_fp64."""
    pos = lattice(box, 61)
    rng = np.random.default_rng(62)
    rc = cutoffs(pos, box, "ramp", rng).astype(np.float32).astype(np.float64)
    for k in rng.choice(np.flatnonzero(rc > 5.9), outside, replace=False):  # in the vapor: nobody on top of another
        d = rng.integers(0, 2)
        pos[k, d] = rng.choice([-0.25, box[d], box[d] + 0.75])
    n = len(pos)
    assert n > 49152
    types = rng.integers(0, ntypes, n).astype(np.float32)
    A = np.concatenate([rng.normal(size=(n, 3)), np.zeros((n, 1))], 1).astype(np.float32)
    res = []
    for prec, real in ((D.DCM_PREC_FP64, torch.float64), (D.DCM_PREC_MIXED, torch.float32)):
        ctx = D.Context(D.make_params(box, n_max=n, ntypes=ntypes, eps=(1.0, 0.8)[:ntypes], sigma=(1.0, 1.1)[:ntypes],
                                      shift_energy=1, precision=prec))
        i32 = dict(dtype=torch.int32, device="cuda")
        cell, start, perm = torch.empty(n, **i32), torch.empty(ctx.ncell + 1, **i32), torch.empty(n, **i32)
        p4 = D.to_real4(torch.from_numpy(pos), torch.from_numpy(types), real)
        ps = torch.empty_like(p4)
        D.dcm_bin(ctx, n, p4, cell, start, perm, ps)
        perm = perm.long()
        G, dpar = torch.full_like(ps, 7.0), torch.full((2 * ntypes,), 7.0, dtype=torch.float64, device="cuda")
        D.dcm_forces_backward(ctx, n, ps, torch.from_numpy(rc).to(real).cuda()[perm].contiguous(), start,
                              torch.from_numpy(A).to(real).cuda()[perm].contiguous(), 0.7, G, dpar)
        out = torch.empty_like(G)
        out[perm] = G
        assert D.dcm_status(ctx) == D.DCM_OK
        res.append((out.double().cpu().numpy(), dpar.cpu().numpy()))
        ctx.close()
    (G0, d0), (G1, d1) = res
    assert np.sqrt(((G1 - G0)[:, :3] ** 2).mean()) <= 5e-6 * np.sqrt((G0[:, :3] ** 2).mean())
    assert np.all(G1[:, 3] == 0.0)
    assert np.all(np.abs(d1 - d0) <= 5e-6 * np.abs(d0).max())


@pytest.mark.parametrize("l", [3.0, 6.0])
@pytest.mark.parametrize("typed", [False, True])
@pytest.mark.parametrize("n,kernel", [(20480, 0), (23552, 3)])
def test_wide_cells_on_both_sides_of_the_switch(D, l, typed, n, kernel):
    """With cells no narrower than rc_min, up to 20,480 particles run 16 lanes
    per particle, one more runs tiles (AUTO); without tiles (PACKED) up to 23,552
    do, and one more runs one thread per particle."""
    box = (60.0, 48.0, 48.0)
    pos = lattice(box, 81, spacing=1.3)
    rng = np.random.default_rng(82)
    pos = pos[np.abs(pos[:, 2] - 24.0) < 12.0]
    pos = pos[rng.permutation(len(pos))]
    assert len(pos) > n
    pos = np.concatenate([pos[:n], [[30.0, 24.0, 1.0]]]).astype(np.float32)
    rc = np.append(np.clip(6.0 - (12.0 - np.abs(pos[:n, 2] - 24.0)), 3.0, 6.0), 6.0)
    types = rng.integers(0, 2 if typed else 1, n + 1).astype(np.float32)
    F0, _ = by_input(D, box, pos[:n], rc[:n], types[:n], l=l, h=1.5, force_kernel=kernel)
    F1, _ = by_input(D, box, pos, rc, types, l=l, h=1.5, force_kernel=kernel)
    assert np.all(F1[n] == 0.0)
    if kernel == D.DCM_FORCE_PACKED:
        assert np.array_equal(F1[:n], F0)  # the same sums in the same order
    assert np.sqrt(((F1[:n] - F0)[:, :3] ** 2).mean()) <= MIXED_RMS * np.sqrt((F0[:, :3] ** 2).mean())
    F0n, t0 = forces(D, box, pos, rc, types if typed else None, force_kernel=D.DCM_FORCE_THREAD, l=l, h=1.5,
                     **(dict(ntypes=2, eps=(1.0, 0.8), sigma=(1.0, 1.1)) if typed else {}))
    F1n, t1 = forces(D, box, pos, rc, types if typed else None, l=l, h=1.5, force_kernel=kernel,
                     **(dict(ntypes=2, eps=(1.0, 0.8), sigma=(1.0, 1.1)) if typed else {}))
    assert t1[2] == t0[2]


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("box,lx,outside", [
    ((480.0, 24.0, 27.0), 0.0, 0),
    ((480.0, 24.0, 27.0), 0.5, 0),    # a last piece of fewer cells
    ((480.0, 24.0, 27.0), 0.75, 1),   # one piece with a coordinate outside the box
    ((600.0, 30.0, 33.0), 1.5, 3),
])
def test_tiles_of_long_bundles(D, box, lx, outside, prec):
    """Few and long bundles of cell rows, which are cut into pieces."""
    pos = lattice(box, 91)
    rng = np.random.default_rng(92)
    for k in rng.choice(np.flatnonzero(np.abs(pos[:, 2] - 0.5 * box[2]) > 0.3 * box[2]), outside, replace=False):
        pos[k, 0] = rng.choice([-0.25, box[0]])
    rc = cutoffs(pos, box, "ramp", rng)
    assert len(pos) > 32768
    walk = D.DCM_FORCE_PACKED if prec == "mixed" else D.DCM_FORCE_THREAD
    F0, t0 = forces(D, box, pos, rc, prec=prec, force_kernel=walk, lx=lx)
    F1, t1 = forces(D, box, pos, rc, prec=prec, lx=lx)
    assert t1[2] == t0[2]
    tol = MIXED_RMS if prec == "mixed" else FP64_RMS
    assert np.sqrt(((F1 - F0)[:, :3] ** 2).mean()) <= tol * np.sqrt((F0[:, :3] ** 2).mean())
    assert abs(t1[0] - t0[0]) <= 4 * tol * np.abs(F0[:, 3]).sum()


def test_lists_and_adjoint_of_long_bundles(D):
    box = (480.0, 33.0, 34.5)
    pos = lattice(box, 93)
    rng = np.random.default_rng(94)
    res = []
    for skin in (0.5, 0.0):
        ctx = D.Context(D.make_params(box, n_max=len(pos), skin=skin, lx=0.5))
        st = D.State(ctx, D.to_real4(torch.from_numpy(pos)), torch.zeros(len(pos), 4))
        D.dcm_step_init(ctx, st)
        assert D.dcm_status(ctx) == D.DCM_OK
        ids = st.current()[3].cpu().numpy()
        F = np.empty((len(pos), 3))
        F[ids] = st.force.double().cpu().numpy()[:, :3]
        res.append((F, st.thermo.cpu().numpy()))
        ctx.close()
    (F0, t0), (F1, t1) = res
    assert t0[3] == t1[3]
    assert np.sqrt(((F0 - F1) ** 2).mean()) <= 1e-5 * np.sqrt((F1 ** 2).mean())
    types = rng.integers(0, 2, len(pos)).astype(np.float32)  # bounds as in test_adjoint_forms_against_fp64
    A = np.concatenate([rng.normal(size=(len(pos), 3)), np.zeros((len(pos), 1))], 1).astype(np.float32)
    rc = cutoffs(pos, box, "ramp", rng).astype(np.float32).astype(np.float64)
    assert len(pos) > 49152
    G0, d0 = by_input(D, box, pos, rc, types, A, lx=0.5, precision=D.DCM_PREC_FP64)
    G1, d1 = by_input(D, box, pos, rc, types, A, lx=0.5)
    assert np.sqrt(((G1 - G0)[:, :3] ** 2).mean()) <= 5e-6 * np.sqrt((G0[:, :3] ** 2).mean())
    assert np.all(np.abs(d1 - d0) <= 5e-6 * np.abs(d0).max())


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n_max", [0, 1_300_000])
def test_long_tiles(D, n_max, prec):
    """A thin gas in a long box: tiles end at their longest (12 rc_max, and 24 in
    contexts of more than 1.2M particles), far from full."""
    box = (450.0, 60.0, 60.0)
    rng = np.random.default_rng(95)
    n = 36000
    pos = (rng.random((n, 3)) * np.array(box)).astype(np.float32)
    pos = np.minimum(pos, np.nextafter(np.array(box, np.float32), np.float32(0)))
    rc = rng.choice([3.0, 6.0], n)
    res = []
    real = torch.float32 if prec == "mixed" else torch.float64
    for kernel in (D.DCM_FORCE_THREAD, D.DCM_FORCE_AUTO):
        ctx = D.Context(D.make_params(box, n_max=max(n, n_max), lx=0.5, force_kernel=kernel,
                                      precision=D.DCM_PREC_MIXED if prec == "mixed" else D.DCM_PREC_FP64))
        p4 = D.to_real4(torch.from_numpy(pos), None, real)
        i32 = dict(dtype=torch.int32, device="cuda")
        cell, start, perm = torch.empty(n, **i32), torch.empty(ctx.ncell + 1, **i32), torch.empty(n, **i32)
        ps = torch.empty_like(p4)
        D.dcm_bin(ctx, n, p4, cell, start, perm, ps)
        F, tot = torch.empty_like(ps), torch.zeros(3, dtype=torch.float64, device="cuda")
        D.dcm_forces(ctx, n, ps, torch.from_numpy(rc).to(real).cuda()[perm.long()].contiguous(), start, F, tot)
        assert D.dcm_status(ctx) == D.DCM_OK
        res.append((F.double().cpu().numpy(), tot.cpu().numpy()))
        ctx.close()
    (F0, t0), (F1, t1) = res
    assert t0[2] == t1[2]
    mag = np.sqrt((F0[:, :3] ** 2).sum(1))  # overlapping particles: each against its own force
    close = np.abs(F1 - F0)[:, :3].max(1) <= (2e-5 if prec == "mixed" else 1e-11) * np.maximum(mag, np.median(mag))
    assert close.all()


@pytest.mark.parametrize("n,same", [(36000, True), (52000, False)])
def test_thin_gas_in_wide_cells(D, n, same):
    """Below 3 particles per sphere of rc_min (26.5 per 1000 sigma^3) AUTO is
    the row walk, with its sums bit for bit; above it runs tiles."""
    box = (120.0, 120.0, 114.0)
    rng = np.random.default_rng(97)
    g = np.stack(np.meshgrid(*[(np.arange(60) + 0.5) * (L / 60) for L in box], indexing="ij"), -1).reshape(-1, 3)
    pos = (g + rng.uniform(-0.4, 0.4, g.shape))[rng.permutation(len(g))[:n]].astype(np.float32)
    rc = np.full(n, 6.0)
    F0, t0 = forces(D, box, pos, rc, l=3.0, h=1.5, force_kernel=D.DCM_FORCE_PACKED)
    F1, t1 = forces(D, box, pos, rc, l=3.0, h=1.5)
    assert t1[2] == t0[2]
    assert np.array_equal(F1, F0) == same
    assert np.sqrt(((F1 - F0)[:, :3] ** 2).mean()) <= MIXED_RMS * np.sqrt((F0[:, :3] ** 2).mean())


@pytest.mark.parametrize("box", [(18.0, 21.0, 24.0), (24.0, 24.0, 120.0)])
@pytest.mark.parametrize("typed,kw", [(False, dict()), (True, dict(newton3=1)), (False, dict(newton3=1, lx=0.5)),
                                      (True, dict(lx=0.75))])
def test_lists_by_the_row_walk(D, box, typed, kw):
    """Boxes of less than 5 (rc_max + skin): full and half lists of the row walk."""
    test_lists_over_tiles(D, box, None, 1.12, typed, kw)


@pytest.mark.parametrize("skin", [0.0, 0.5])
def test_adjoint_between_steps(D, skin):
    """The tiled adjoint keeps its records in the binning's scratch: steps
    around it give what they give without it, and it gives the same twice."""
    box = (63.0, 61.5, 72.0)
    pos = lattice(box, 98)
    n = len(pos)
    assert n > 49152
    rng = np.random.default_rng(99)
    vel = torch.from_numpy(rng.normal(size=(n, 4)).astype(np.float32))
    vel[:, 3] = 0
    A = torch.from_numpy(rng.normal(size=(n, 4)).astype(np.float32)).cuda()
    i32 = dict(dtype=torch.int32, device="cuda")
    res, grads = [], []
    for adjoint in (False, True):
        ctx = D.Context(D.make_params(box, n_max=n, skin=skin, recompute_every=3))
        st = D.State(ctx, D.to_real4(torch.from_numpy(pos)), vel)
        D.dcm_step_init(ctx, st)
        p4 = D.to_real4(torch.from_numpy(pos))
        cell, start, perm = torch.empty(n, **i32), torch.empty(ctx.ncell + 1, **i32), torch.empty(n, **i32)
        ps = torch.empty_like(p4)
        D.dcm_bin(ctx, n, p4, cell, start, perm, ps)
        rc = torch.full((n,), 3.5, device="cuda")
        for k in range(4):
            if adjoint:
                G, d = torch.empty_like(ps), torch.empty(2, dtype=torch.float64, device="cuda")
                D.dcm_forces_backward(ctx, n, ps, rc, start, A, 0.7, G, d)
                grads.append((G.cpu(), d.cpu()))
            D.dcm_step(ctx, st, 0.002, 2)
        assert D.dcm_status(ctx) == D.DCM_OK
        res.append([t.cpu() for t in st.current()] + [st.force.cpu()])
        ctx.close()
    for a, b in zip(*res):
        assert torch.equal(a, b)
    for G, d in grads[1:]:
        assert torch.equal(G, grads[0][0]) and torch.allclose(d, grads[0][1], rtol=1e-12, atol=0)


@pytest.mark.parametrize("n,box,kw,name", [
    (2000, (12.0, 12.0, 48.0), dict(), "k_forces_planes"),
    (32768, (61.5, 61.5, 61.5), dict(), "k_forces_planes"),
    (32769, (61.5, 61.5, 61.5), dict(), "k_forces_tiles"),
    (32769, (22.5, 61.5, 61.5), dict(), "k_forces_x2"),              # narrower than 4 rc_max
    (32769, (61.5, 61.5, 61.5), dict(force_kernel=3), "k_forces_x2"),
    (32769, (61.5, 61.5, 61.5), dict(accumulation=1), "k_forces_x2"),
    (2000, (12.0, 12.0, 48.0), dict(force_kernel=1), "k_forces"),
    (32769, (61.5, 61.5, 61.5), dict(ntypes=3, eps=(1, 1, 1), sigma=(1, 1, 1)), "k_forces"),
    (20480, (60.0, 60.0, 60.0), dict(l=3.0, h=1.5), "k_forces_planes"),
    (20481, (60.0, 60.0, 60.0), dict(l=3.0, h=1.5), "k_forces_tiles"),
    (23553, (60.0, 60.0, 60.0), dict(l=3.0, h=1.5, force_kernel=3), "k_forces_x2"),
    (3999, (24.0, 24.0, 48.0), dict(precision=0), "k_forces"),
    (4000, (24.0, 24.0, 48.0), dict(precision=0), "k_forces_tiles"),
])
def test_force_search(D, n, box, kw, name):
    """Which kernel a force launch of n particles runs."""
    ctx = D.Context(D.make_params(box, n_max=40000, **kw))
    assert D.force_kernel_name(ctx, n) == name
    ctx.close()
