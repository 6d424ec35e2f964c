"""Grid stages at the edges of their tiles: blocks of 32 x 8 columns that march
along z (box sums, segmentation, first distance sweep), rows of a multiple of
four boxes or not, half widths beyond the fused box sum, cells of many
particles in the placement.

Integers are compared bit for bit with the oracle.  Distances: |dD| <= 1e-5
max(D, h) (the parity tolerance: a chain of at most ten FP32 updates of a few
ulps each).
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import paper_1701_05242_gb300.dcm as dcm
    return dcm


def context(D, nh, **kw):
    return D.Context(D.make_params(tuple(1.5 * k for k in nh), n_max=16, rc_min=1.5, rc_max=1.5, **kw))


@pytest.mark.parametrize("nh", [(33, 9, 70), (32, 8, 64), (31, 7, 3), (3, 2, 5), (64, 17, 131)])
@pytest.mark.parametrize("w", [0, 1, 2, 3, 4, 5])
def test_box_sums_and_segmentation(D, nh, w):
    rng = np.random.default_rng(100 * w + nh[0])
    nb = int(np.prod(nh))
    count = rng.poisson(1.5, nb).astype(np.int32)
    count.reshape(nh[::-1])[: nh[2] // 2] += 4
    ctx = context(D, nh, smooth_w=w)
    dev = dict(device="cuda")
    s, iface = torch.empty(nb, dtype=torch.uint8, **dev), torch.empty(nb, dtype=torch.uint8, **dev)
    T, g = torch.empty(1, dtype=torch.int32, **dev), torch.empty(nb, dtype=torch.int32, **dev)
    D.dcm_detect_interface(ctx, torch.from_numpy(count).cuda(), s, iface, T, g)
    og, oT, os_, oif = O.detect_interface(count, np.array(nh), w)
    assert np.array_equal(g.cpu().numpy(), og)
    assert int(T.item()) == oT
    assert np.array_equal(s.cpu().numpy(), os_) and np.array_equal(iface.cpu().numpy(), oif)
    assert D.dcm_status(ctx) == D.DCM_OK


@pytest.mark.parametrize("nh", [(32, 9, 33), (36, 8, 5), (35, 11, 7), (4, 3, 40), (2, 2, 2)])
def test_distances(D, nh):
    rng = np.random.default_rng(nh[0])
    nb = int(np.prod(nh))
    s = np.ones(nb, np.uint8)
    iface = (rng.random(nb) < 0.01).astype(np.uint8)
    iface[0] = 1
    s[rng.random(nb) < 0.005] = 0
    ctx = context(D, nh, r_grid=7.5)
    Dg = torch.empty(nb, dtype=torch.float32, device="cuda")
    D.dcm_distance(ctx, torch.from_numpy(s).cuda(), torch.from_numpy(iface).cuda(), Dg)
    Dj, _ = O.distance_jacobi(s, iface, np.array(nh), 1.5, 7.5)
    Dg = Dg.cpu().numpy().astype(np.float64)
    fin = np.isfinite(Dj) & np.isfinite(Dg)
    other = np.where(np.isfinite(Dj), Dj, Dg)[np.isfinite(Dj) != np.isfinite(Dg)]
    assert np.all(other >= 7.5 * (1 - 1e-5))  # FP32 and FP64 may round the threshold apart
    assert np.all(np.abs(Dg[fin] - Dj[fin]) <= 1e-5 * np.maximum(Dj[fin], 1.5))


@pytest.mark.parametrize("n", [1, 31, 257, 5000])
def test_placement_of_crowded_cells(D, n):
    """Most particles in three cells, in no order: the stable order is exact."""
    rng = np.random.default_rng(n)
    box = (6.0, 9.0, 12.0)
    pos = rng.random((n, 3)) * np.array(box)
    crowd = rng.random(n) < 0.8
    pos[crowd] = np.array([[0.2, 0.3, 0.4], [5.9, 8.9, 11.9], [3.1, 4.6, 6.1]])[rng.integers(0, 3, crowd.sum())]
    pos = np.minimum(pos, np.nextafter(np.array(box, np.float32), np.float32(0))).astype(np.float32)
    ctx = D.Context(D.make_params(box, n_max=n, rc_min=1.5, rc_max=3.0))
    p4 = D.to_real4(torch.from_numpy(pos))
    i32 = dict(dtype=torch.int32, device="cuda")
    cell, start, perm = torch.empty(n, **i32), torch.empty(ctx.ncell + 1, **i32), torch.empty(n, **i32)
    ps = torch.empty_like(p4)
    D.dcm_bin(ctx, n, p4, cell, start, perm, ps)
    oc, _, ostart, operm = O.bin_particles(pos, box, 1.5)
    assert np.array_equal(cell.cpu().numpy(), oc) and np.array_equal(start.cpu().numpy(), ostart)
    assert np.array_equal(perm.cpu().numpy(), operm)
    assert np.array_equal(ps.cpu().numpy(), p4.cpu().numpy()[operm])


def test_distances_with_an_exhausted_wait_budget(D):
    """A wait budget of 1 microsecond, below the time between the first and the
    last block of a sweep: the launch ends, and the call says so instead of
    returning unfinished distances; with the budget restored it gives what a fresh
    context gives."""
    nh = (96, 96, 96)
    nb = int(np.prod(nh))
    rng = np.random.default_rng(1)
    s = torch.ones(nb, dtype=torch.uint8, device="cuda")
    iface = torch.from_numpy((rng.random(nb) < 0.002).astype(np.uint8)).cuda()
    i32 = dict(dtype=torch.int32, device="cuda")

    def run(ctx):
        d, it = torch.empty(nb, device="cuda"), torch.full((1,), 77, **i32)
        try:
            D.dcm_distance(ctx, s, iface, d, it)
            code = D.DCM_OK
        except D.DcmError as e:
            code = e.code
        return code, d, int(it.item())

    ctx, fresh = context(D, nh, r_grid=12.0), context(D, nh, r_grid=12.0)
    code, d0, it0 = run(fresh)
    assert code == D.DCM_OK and it0 > 5
    with pytest.raises(D.DcmError):
        D.dcm_set_wait_budget(ctx, 999)
    D.dcm_set_wait_budget(ctx, 1000)
    code, _, it = run(ctx)
    assert code == D.DCM_ERR_TIMEOUT and it == -1
    assert D.dcm_status(ctx) == D.DCM_ERR_TIMEOUT
    D.dcm_set_wait_budget(ctx, 2_000_000_000)
    code, d, it = run(ctx)
    assert code == D.DCM_OK and it == it0 and torch.equal(d, d0)
    assert D.dcm_status(ctx) == D.DCM_OK
