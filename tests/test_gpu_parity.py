"""Parity of the CUDA path with the CPU oracle, through the C interface.

Connectivity (vertex ids of every triangle, in the canonical order), labels
and pattern codes must be bit-exact; coordinates agree within 1e-6 h.  Small
cases compare every intermediate stage too (segments, grid-edge events and
their vertex ids, per-cell records)."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same_mesh, gpu_mesh
from mesh_checks import check_mesh
from paper_2602_19474_gb300 import synth

pytestmark = pytest.mark.gpu


def run_both(img, hn, hd=1, stages=True, on_device=False):
    g = gpu_mesh(img, hn, hd, stages=stages, on_device=on_device)
    o = oracle.mesh_bitmap(img, hn, hd)
    assert_same_mesh(g, o, hn / hd, W=img.shape[1], stages=stages)
    return g, o


def test_disk64_h2():
    g, o = run_both(synth.disk(), 2)
    check_mesh(synth.disk(), g["xy"], g["tri"], g["label"], 2.0, g["n_cells"])


@pytest.mark.parametrize("hn,hd", [(2, 1), (4, 1), (8, 1), (2, 3), (4, 7), (6, 5)])
def test_disk_grid_sizes(hn, hd):
    run_both(synth.disk(size=40, cx=19, cy=21, r=13), hn, hd)


def test_constant_and_tiny_images():
    run_both(np.full((5, 7), 9, np.uint8), 2)
    run_both(np.zeros((1, 1), np.uint8), 2)
    run_both(np.ones((1, 37), np.uint8), 4)
    run_both(np.ones((29, 1), np.uint16), 2)


def test_every_3x3_bitmap_h2():
    for bits in range(0, 512, 7):
        img = np.array([(bits >> k) & 1 for k in range(9)], np.uint8).reshape(3, 3)
        run_both(img, 2)


def test_multilabel_u16_and_junctions():
    rng = np.random.default_rng(11)
    for _ in range(10):
        img = rng.integers(0, 4, (9, 13)).astype(np.uint16) * 1000
        run_both(img, 2)
        run_both(img, 8)
    v = synth.voronoi_labels(size=200, nseeds=60, nlabels=16)
    run_both(v, 2)


def test_checkerboard_pinches_and_islands():
    cb = (np.indices((17, 23)).sum(axis=0) % 2).astype(np.uint8)
    run_both(cb, 2)
    run_both(cb, 8)
    isl = np.zeros((60, 70), np.uint8)
    isl[5::9, 7::11] = 1
    isl[30:33, 30:33] = 2
    run_both(isl, 8)


def test_noise_bitmaps_all_h():
    for k, img in enumerate(synth.noise_batch(n=6, lo=50, hi=300, first=6)):
        for hn in (2, 4, 8):
            run_both(img, hn, stages=(k < 2))


def test_device_resident_input_matches_host_input():
    img = synth.ellipses(size=300, n=20, amin=8, amax=60)
    a = gpu_mesh(img, 4, stages=False)
    b = gpu_mesh(img, 4, stages=False, on_device=True)
    for k in ("tri", "label", "code"):
        assert np.array_equal(a[k], b[k])
    assert np.array_equal(a["xy"], b["xy"])


def test_ellipses2048_full_size():
    img = synth.ellipses()
    g, o = run_both(img, 4, stages=False)
    check_mesh(img, g["xy"], g["tri"], g["label"], 4.0, g["n_cells"])


def test_paper_regime_no_tier_g():
    img = synth.disk(size=48, cx=24, cy=24, r=15)
    g, o = run_both(img, 2, 3)
    assert g["n_tierG_cells"] == 0


def test_voronoi8192_full_size():
    """The 8192^2 16-label workload in the bench's launch configuration
    (device-resident u16 image, h = 2) against the oracle's mesh of the whole
    image: every triangle's vertex ids, label and code bit-exact, every
    coordinate within 1e-6 h, plus the exact area identities."""
    from gpu_util import exact_area_checks

    img = synth.voronoi_labels()
    g = gpu_mesh(img, 2, 1, on_device=True)
    o = oracle.mesh_bitmap(img, 2, 1)
    assert_same_mesh(g, o, 2.0, W=img.shape[1])
    exact_area_checks(img, g, 2.0)


def test_serving_pool_images_all_h():
    """Serving-pool bitmaps (square thresholded noise, sides up to 4057 px):
    the largest one at h = 2, 4 and 8, and three more at their own h, each
    against the oracle in full."""
    specs = synth.serving_specs()
    order = sorted(range(len(specs)), key=lambda i: specs[i][0])
    big = specs[order[-1]]
    img = synth.serving_image(big)
    for hn in (4, 8, 2):
        run_both(img, hn, stages=False)
    for k in (order[len(order) // 4], order[len(order) // 2], order[(3 * len(order)) // 4]):
        run_both(synth.serving_image(specs[k]), specs[k][2], stages=False)


@pytest.mark.parametrize("seed,h,sigma,sizes", [
    (0, 4, 1.0, (7, 8, 9, 16, 17)),
    (0, 8, 1.5, (8, 9, 16, 17)),
    (0, 14, 2.0, (8, 9, 16, 17, 32, 33, 37)),
])
def test_tier_g_cells_of_every_group_size(seed, h, sigma, sizes):
    """Tier-G cells of as many vertices as a group of 8, 16 or 32 lanes takes,
    and of one more (the list form above 32): the mesh is the oracle's."""
    img = synth.noise_bitmap(np.random.default_rng(seed), 260, 230, sigma)
    g, o = run_both(img, h)
    cut = o["cut"][o["cut"][:, 4] == 1]
    have = set((cut[:, 2] + 2 - cut[:, 3]).tolist())
    assert have.issuperset(sizes), sorted(have)


@pytest.mark.parametrize("hn,hd", [(2, 1), (4, 1), (2, 3)])
def test_irrational_event_coordinates_to_the_bit(hn, hd):
    """An event's irrational coordinate is (a + b sqrt3) / S with whole a, b and S
    = 6 h_den: one rounding for the sum (with the double next to sqrt3), one for the
    product with 1 / S."""
    from fractions import Fraction

    import paper_2602_19474_gb300 as sb
    from gpu_util import ctx

    img = synth.voronoi_labels(size=48, nseeds=9)
    c = ctx()
    m = sb.mesh_bitmap(c, img, hn, hd)
    xy = sb.view_numpy(sb.mesh_query(c, m, -1))["xy"].copy()
    sb.mesh_release(c, m)
    S, r3 = 6 * hd, 1.7320508075688772935
    b = np.arange(-200 * hd, 200 * hd + 1)
    b = b[b != 0]
    seen = 0
    for x in xy[:, 0]:
        if abs(x * S - round(x * S)) < 1e-6:
            continue
        a = np.rint(x * S - b * r3)
        d = np.abs(a + b * r3 - x * S)
        k = int(d.argmin())
        assert d[k] < 1e-9
        assert float(Fraction(int(a[k])) + Fraction(int(b[k])) * Fraction(r3)) * (1.0 / S) == x
        seen += 1
    assert seen > 100
