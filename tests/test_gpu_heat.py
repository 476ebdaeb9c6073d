"""mesh_heat (App. H) on the device against the heat-diffusion oracle on the
same mesh: the solution after several backward-Euler steps and the peak per
step.  The device solves each step by conjugate gradients to a relative
residual of 1e-12 and sums in a different order, so the two agree to a
tolerance of 1e-8 of the pulse's amplitude rather than bit for bit.  At
full size the device's solution is checked against the oracle's operator:
the residual of the backward-Euler equation of its first step."""
import numpy as np
import pytest

import oracle
import paper_2602_19474_gb300 as sb
from gpu_util import ctx
from oracle import heat as H
from paper_2602_19474_gb300 import synth

pytestmark = pytest.mark.gpu


def run_gpu(m, L, alpha, dt, steps, x0, y0, sigma, amp=100.0, tol=1e-12):
    u, peaks, its = sb.mesh_heat(ctx(), m, L, alpha, dt, steps, x0, y0, sigma, amp, tol)
    return u.cpu().numpy(), np.array(peaks), its


CASES = [
    # image, h, label, alpha, dt, steps, pulse centre and width
    ("rectangle", lambda: np.pad(np.ones((40, 60), np.uint8), 10), 2, 1, 1, 500.0, 0.01, 5, (40.0, 30.0), 15.0),
    ("voronoi", lambda: synth.voronoi_labels(size=128, nseeds=12), 2, 1, None, 50.0, 0.05, 4, (64.0, 64.0), 20.0),
    ("voronoi_fine", lambda: synth.voronoi_labels(size=64, nseeds=6), 2, 3, None, 20.0, 0.05, 3, (30.0, 34.0), 10.0),
    ("disk", lambda: synth.disk(), 2, 1, 1, 100.0, 0.02, 6, (31.5, 31.5), 12.0),
]


@pytest.mark.parametrize("name,make,hn,hd,L,alpha,dt,steps,c,sigma", CASES, ids=[c[0] for c in CASES])
def test_parity_with_oracle(name, make, hn, hd, L, alpha, dt, steps, c, sigma):
    img = make()
    if L is None:
        L = int(np.bincount(img.ravel()).argmax())
    cx = ctx()
    m = sb.mesh_bitmap(cx, img, hn, hd)
    g = sb.view_numpy(sb.mesh_query(cx, m, -1))
    u, peaks, its = run_gpu(m, L, alpha, dt, steps, c[0], c[1], sigma)
    sb.mesh_release(cx, m)
    uo, po = H.heat(g["xy"], g["tri"], g["label"], L, alpha, dt, steps, c[0], c[1], sigma)
    assert np.abs(u - uo).max() <= 1e-8 * 100.0, np.abs(u - uo).max()
    assert np.allclose(peaks, po, rtol=0, atol=1e-8 * 100.0)
    assert all(0 < k < 10000 for k in its)
    _, free, _ = H.region(g["tri"], g["label"], L)
    assert (u[~free] == 0).all()


def test_on_the_preprocessed_mesh():
    img = synth.voronoi_labels(size=96, nseeds=10)
    L = int(np.bincount(img.ravel()).argmax())
    cx = ctx()
    m = sb.mesh_preprocess(cx, img, 2, 1)
    g = sb.view_numpy(sb.mesh_query(cx, m, -1))
    u, peaks, _ = run_gpu(m, L, 30.0, 0.05, 3, 48.0, 48.0, 15.0)
    sb.mesh_release(cx, m)
    uo, po = H.heat(g["xy"], g["tri"], g["label"], L, 30.0, 0.05, 3, 48.0, 48.0, 15.0)
    assert np.abs(u - uo).max() <= 1e-6, np.abs(u - uo).max()


def test_bad_parameters_and_no_convergence():
    cx = ctx()
    m = sb.mesh_bitmap(cx, synth.disk(), 2, 1)
    with pytest.raises(sb.SbmtError) as e:
        sb.mesh_heat(cx, m, 1, 100.0, -1.0, 2, 0.0, 0.0, 5.0)
    assert e.value.code == sb.SBMT_EINVAL
    with pytest.raises(sb.SbmtError) as e:  # one iteration cannot reach 1e-14
        sb.mesh_heat(cx, m, 1, 100.0, 0.05, 1, 31.5, 31.5, 12.0, tol=1e-14, max_iterations=1)
    assert e.value.code == sb.SBMT_ETIMEDOUT
    # a label with no triangles: nothing is free, u stays 0
    u, peaks, its = sb.mesh_heat(cx, m, 77, 100.0, 0.05, 2, 31.5, 31.5, 12.0)
    assert float(u.abs().max()) == 0.0 and peaks == [0.0, 0.0] and its == [0, 0]
    sb.mesh_release(cx, m)


def test_full_size_residual():
    """voronoi8192's mesh (8192^2 u16, h = 2), the most frequent label: the
    device's first step satisfies the oracle's backward-Euler equation to the
    solver's tolerance."""
    import scipy.sparse as sp

    img = synth.voronoi_labels()
    L = int(np.bincount(img.ravel()).argmax())
    cx = ctx()
    m = sb.mesh_bitmap(cx, img, 2, 1)
    # host copies of the mesh first: the views die with the mesh
    t = sb.view_tensors(sb.mesh_query(cx, m, -1))
    lab = t["label"].cpu().numpy().view(np.uint16)
    tri_all = t["tri"].cpu().numpy()
    xy = t["xy"].cpu().numpy()
    del t
    tri = tri_all[lab == L]
    alpha, dt, sigma = 500.0, 0.01, 127.0
    u, peaks, its = run_gpu(m, L, alpha, dt, 1, 4096.0, 4096.0, sigma, tol=1e-10)
    sb.mesh_release(cx, m)
    nv = len(xy)
    allsel, free, _ = H.region(tri_all, lab, L)
    K = H.stiffness(xy, tri, nv)
    M = H.lumped_mass(xy, tri, nv)
    u0 = np.where(free, H.pulse(xy, 4096.0, 4096.0, sigma, 100.0), 0.0)
    res = (sp.diags(M) @ u + alpha * dt * (K @ u) - M * u0)[free]
    rhs = (M * u0)[free]
    assert np.linalg.norm(res) <= 2e-10 * np.linalg.norm(rhs), np.linalg.norm(res) / np.linalg.norm(rhs)
    assert free.sum() > 100000 and 0 < peaks[0] <= 100.0


def test_runs_are_bit_identical():
    """The assembly and the solver's reductions sum in fixed orders (records
    placed by a scan, each vertex's mass and diagonal gathered in record
    order, rows sorted by column, block partials added in block order), so
    two runs give the same bits."""
    img = synth.voronoi_labels(size=700, nseeds=40)
    L = int(np.bincount(img.ravel()).argmax())
    cx = ctx()
    m = sb.mesh_bitmap(cx, img, 2, 1)
    a = run_gpu(m, L, 500.0, 0.01, 4, 350.0, 350.0, 60.0)
    b = run_gpu(m, L, 500.0, 0.01, 4, 350.0, 350.0, 60.0)
    sb.mesh_release(cx, m)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2]


@pytest.mark.parametrize("side,fan", [(3, 9), (21, 40), (22, 7), (23, 200), (120, 33)])
def test_block_edges_and_long_rows(side, fan):
    """Regions of one block (22^2 + fan - 1 vertices: 484 + 7 = 491), just over
    one, and many, each with a vertex of `fan` neighbours (a row beyond the
    eight entries kept in slices): an imported square grid and a fan apart from
    it, every vertex free.  Tolerance as in test_parity_with_oracle."""
    j, i = np.mgrid[0:side, 0:side]
    xy = np.stack([i.ravel(), j.ravel() * 0.9], 1).astype(float)
    a = (j[:-1, :-1] * side + i[:-1, :-1]).ravel()
    tri = np.concatenate([np.stack([a, a + 1, a + side + 1], 1), np.stack([a, a + side + 1, a + side], 1)])
    n = len(xy)
    ang = 2 * np.pi * np.arange(fan) / fan
    xy = np.concatenate([xy, [[-8.0, -8.0]], np.stack([-8 + 3 * np.cos(ang), -8 + 3 * np.sin(ang)], 1)])
    k = np.arange(fan)
    tri = np.concatenate([tri, np.stack([np.full(fan, n), n + 1 + k, n + 1 + (k + 1) % fan], 1)]).astype(np.int32)
    m = sb.mesh_import(ctx(), xy, tri)
    u, peaks, its = run_gpu(m, 0xFFFF, 3.0, 0.1, 3, 2.0, 1.0, 6.0)
    sb.mesh_release(ctx(), m)
    uo, po = H.heat(xy, tri, np.full(len(tri), 0xFFFF), 0xFFFF, 3.0, 0.1, 3, 2.0, 1.0, 6.0)
    assert np.abs(u - uo).max() <= 1e-8 * 100.0
    assert np.allclose(peaks, po, rtol=0, atol=1e-8 * 100.0)


@pytest.mark.parametrize("side", [831, 832])
def test_vectors_on_chip_and_beyond(side):
    """The largest square grid whose vectors fit the blocks' shared memory (152
    blocks of 4544 rows), and the next one, which keeps them in L2: the first step
    satisfies the oracle's backward-Euler equation.  The solver stops at a relative
    residual of 1e-10; the recurrences drift from the true residual by some 1e-14."""
    import scipy.sparse as sp

    j, i = np.mgrid[0:side, 0:side]
    xy = np.stack([i.ravel(), j.ravel() * 0.9], 1).astype(float)
    a = (j[:-1, :-1] * side + i[:-1, :-1]).ravel()
    tri = np.concatenate([np.stack([a, a + 1, a + side + 1], 1), np.stack([a, a + side + 1, a + side], 1)]).astype(np.int32)
    m = sb.mesh_import(ctx(), xy, tri)
    alpha, dt = 500.0, 0.01
    u, peaks, its = run_gpu(m, 0xFFFF, alpha, dt, 1, 400.0, 380.0, 60.0, tol=1e-10)
    sb.mesh_release(ctx(), m)
    K, M = H.stiffness(xy, tri, len(xy)), H.lumped_mass(xy, tri, len(xy))
    rhs = M * H.pulse(xy, 400.0, 380.0, 60.0, 100.0)
    res = sp.diags(M) @ u + alpha * dt * (K @ u) - rhs
    assert np.linalg.norm(res) <= 2e-10 * np.linalg.norm(rhs), np.linalg.norm(res) / np.linalg.norm(rhs)
    assert 0 < peaks[0] <= 100.0


@pytest.mark.parametrize("amplitude,peak", [(np.nan, 0.0), (np.inf, np.inf), (-np.inf, 0.0)])
def test_peaks_leave_nans_out(amplitude, peak):
    """The peak is the maximum of 0 and the values that are numbers: with an
    amplitude that is none, or where an infinite one meets an exponential that is
    0 (NaN far from the centre), no step iterates and the peak holds no NaN."""
    m = sb.mesh_bitmap(ctx(), synth.disk(), 2, 1)
    u, peaks, its = run_gpu(m, 1, 100.0, 0.05, 2, 31.5, 31.5, 0.5, amp=amplitude)
    sb.mesh_release(ctx(), m)
    assert peaks.tolist() == [peak, peak]
    assert its == [0, 0] and np.isnan(u).any()


@pytest.mark.parametrize("blocks", [1, 2, 7, 151])
def test_fewer_sms(blocks):
    """The solver with as few blocks as a part with fewer SMs has, vectors on
    chip and (one block of 88^2 rows) beyond: the oracle's solution."""
    side = 88
    j, i = np.mgrid[0:side, 0:side]
    xy = np.stack([i.ravel(), j.ravel() * 0.9], 1).astype(float)
    a = (j[:-1, :-1] * side + i[:-1, :-1]).ravel()
    tri = np.concatenate([np.stack([a, a + 1, a + side + 1], 1), np.stack([a, a + side + 1, a + side], 1)]).astype(np.int32)
    m = sb.mesh_import(ctx(), xy, tri)
    sb.mesh_heat_debug(ctx(), sb.SBMT_HEAT_BLOCKS, blocks)
    try:
        u, peaks, its = run_gpu(m, 0xFFFF, 3.0, 0.1, 3, 40.0, 38.0, 9.0)
    finally:
        sb.mesh_heat_debug(ctx(), sb.SBMT_HEAT_BLOCKS, 0)
        sb.mesh_release(ctx(), m)
    uo, po = H.heat(xy, tri, np.full(len(tri), 0xFFFF), 0xFFFF, 3.0, 0.1, 3, 40.0, 38.0, 9.0)
    assert np.abs(u - uo).max() <= 1e-8 * 100.0
    assert np.allclose(peaks, po, rtol=0, atol=1e-8 * 100.0)


@pytest.mark.parametrize("barrier", [1, 2, 5])
def test_a_wait_that_runs_out(barrier):
    """One block withholds its sums at a barrier: the call ends with the bounded
    wait's error, u, peaks and iterations unwritten, and the next call on the
    context is right."""
    import torch

    m = sb.mesh_bitmap(ctx(), np.pad(np.ones((70, 80), np.uint8), 4), 2, 1)
    v = sb.mesh_query(ctx(), m, -1)
    args = (1, 50.0, 0.05, 2, 40.0, 38.0, 12.0)
    u = torch.full((v.n_vertices,), 7.0, dtype=torch.float64, device="cuda")
    sb.mesh_heat_debug(ctx(), sb.SBMT_HEAT_STALL, barrier)
    try:
        with pytest.raises(sb.SbmtError) as e:
            sb.mesh_heat(ctx(), m, *args, 100.0, 1e-12, u=u)
    finally:
        sb.mesh_heat_debug(ctx(), sb.SBMT_HEAT_STALL, 0)
    assert e.value.code == sb.SBMT_ETIMEDOUT and "device wait" in str(e.value)
    assert bool((u == 7.0).all())
    got, peaks, its = run_gpu(m, *args)
    g = sb.view_numpy(v)
    sb.mesh_release(ctx(), m)
    uo, po = H.heat(g["xy"], g["tri"], g["label"], *args)
    assert np.abs(got - uo).max() <= 1e-8 * 100.0 and np.allclose(peaks, po, rtol=0, atol=1e-8 * 100.0)


@pytest.mark.parametrize("alpha_dt", [500.0, 5.0e4, 5.0e6])
def test_reachable_residual_at_long_steps(alpha_dt):
    """Steps far longer than a cell's diffusion time (hundreds of iterations):
    the true residual that a step ends at, with a tolerance below what can be
    reached, is no larger than that of conjugate gradients whose every q is the
    product A p, as the geometric mean over 16 pulses (one pulse's ratio moves by
    a few tenths with the rounding)."""
    import scipy.sparse as sp

    img = synth.voronoi_labels(size=200, nseeds=5)
    L = int(np.bincount(img.ravel()).argmax())
    m = sb.mesh_bitmap(ctx(), img, 2, 1)
    g = sb.view_numpy(sb.mesh_query(ctx(), m, -1))
    sel, free, _ = H.region(g["tri"], g["label"], L)
    idx, t = np.nonzero(free)[0], g["tri"][sel]
    M = H.lumped_mass(g["xy"], t, len(g["xy"]))[idx]
    A = (H.stiffness(g["xy"], t, len(g["xy"])) * alpha_dt)[idx][:, idx].tocsr() + sp.diags(M).tocsr()
    P = g["xy"][idx]
    rng = np.random.default_rng(11)
    log = []
    for _ in range(16):
        c = P.mean(0) + np.ptp(P, axis=0) * rng.uniform(-0.25, 0.25, 2)
        sigma = rng.uniform(5.0, 20.0)
        u, _, _ = run_gpu(m, L, alpha_dt, 1.0, 1, c[0], c[1], sigma, tol=1e-13)
        x = H.pulse(P, c[0], c[1], sigma, 100.0)
        b, dinv = M * x, 1.0 / A.diagonal()
        end = np.linalg.norm(b - A @ u[idx])
        r = b - A @ x
        z = r * dinv
        p, rz, it = z.copy(), r @ z, 0
        while it % 8 or np.linalg.norm(r) > 1e-13 * np.linalg.norm(b):
            q = A @ p
            al = rz / (p @ q)
            x, r = x + al * p, r - al * q
            z = r * dinv
            p, rz, it = z + (r @ z) / rz * p, r @ z, it + 1
        log.append(np.log(end / np.linalg.norm(b - A @ x)))
    sb.mesh_release(ctx(), m)
    assert np.mean(log) <= 0.0, np.exp(np.mean(log))


@pytest.mark.parametrize("n", [511, 512, 513, 1024, 1025])
def test_regions_at_the_edges_of_a_block(n):
    """Regions of n free vertices, one block's threads, one more and so on (a fan of
    neighbours around a centre, every vertex free): the oracle's solution."""
    k = np.arange(n - 1)
    ang = 2 * np.pi * k / (n - 1)
    rad = 20.0 + (k % 2)
    xy = np.concatenate([[[0.0, 0.0]], np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1)])
    tri = np.stack([np.zeros(n - 1, int), 1 + k, 1 + (k + 1) % (n - 1)], 1).astype(np.int32)
    m = sb.mesh_import(ctx(), xy, tri)
    u, peaks, its = run_gpu(m, 0xFFFF, 3.0, 0.1, 3, 2.0, 1.0, 9.0)
    sb.mesh_release(ctx(), m)
    uo, po = H.heat(xy, tri, np.full(len(tri), 0xFFFF), 0xFFFF, 3.0, 0.1, 3, 2.0, 1.0, 9.0)
    assert np.abs(u - uo).max() <= 1e-8 * 100.0
    assert np.allclose(peaks, po, rtol=0, atol=1e-8 * 100.0)
