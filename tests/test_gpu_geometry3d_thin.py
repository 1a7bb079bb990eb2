"""Closest features among faces that the FP32 bounds could not judge by their shape or size: hundreds of thin faces (the
angle at a corner below 1e-4), and whole bodies far smaller than 1.  Records bit for bit against the FP64 oracle, and
the search still excludes faces: it may cost a few times the search among other faces, not the evaluation of every face
at every node (20 times and more)."""
import time

import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_geometry3d import _check, ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _fan(verts, tris, face, pieces, depth):
    """The face with its first edge broken into pieces set back by depth of its height, and the thin faces that close
    the surface along the edge."""
    a, b, c = tris[face]
    A, B, C = verts[a], verts[b], verts[c]
    cut = [A + (B - A) * k / pieces + (C - A) * depth for k in range(1, pieces)]
    ids = [a] + [len(verts) + k for k in range(pieces - 1)] + [b]
    fan = [(ids[k], ids[k + 1], c) for k in range(pieces)] + [(a, ids[k + 1], ids[k]) for k in range(1, pieces)]
    return np.concatenate([verts, cut]), np.concatenate([np.delete(tris, face, 0), fan]).astype(np.int32)


def _seconds(ibm, verts, tris, n, lo, hi):  # noqa: F811
    b = ibm.Body3D(verts, tris)
    best = 1e9
    for _ in range(6):
        t = time.perf_counter()
        b.classify(n, lo, hi)
        b.counts()
        best = min(best, time.perf_counter() - t)
    b.close()
    return best


@pytest.mark.parametrize("depth", [0.0, 1e-9, 1e-7, 3e-5])
@pytest.mark.parametrize("pieces", [3, 200])
def test_thin_faces(ibm, orc, depth, pieces):  # noqa: F811
    verts, tris = W.uv_sphere(13, 18, 0.35, (0.503, 0.498, 0.501))
    verts, tris = _fan(verts, tris, 200, pieces, depth)
    _check(ibm, orc, verts, tris, (26, 27, 33), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def test_all_faces_thin(ibm, orc):  # noqa: F811
    verts, tris = W.uv_sphere(2, 120, 0.35, (0.503, 0.498, 0.501))
    verts = verts * [1.0, 1.0, 1e-4] + [0.0, 0.0, 0.5]
    verts, tris = _fan(verts, tris, 7, 40, 1e-8)
    _check(ibm, orc, verts, tris, (26, 27, 33), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def _tube(levels, length):
    """A closed tube of radius 0.35 along z with 6 4^levels sides, its ends closed by rings of a quarter of the vertices
    each: no vertex joins many faces, and the sides of a long tube are thin."""
    verts, tris, rings = [], [], []
    ends = [(k, -0.5) for k in range(levels + 1)] + [(k, 0.5) for k in range(levels, -1, -1)]
    for k, z in ends:
        n = 6 * 4 ** k
        a = 2.0 * np.pi * np.arange(n) / n
        r = 0.35 * (1.0 + k) / (1.0 + levels)
        rings.append((len(verts), n))
        verts += list(np.stack([r * np.cos(a), r * np.sin(a), np.full(n, z * length)], 1))
    for (p, n), (q, m) in zip(rings, rings[1:]):
        for j in range(max(n, m)):
            if n == m:
                tris += [(p + j, p + (j + 1) % n, q + (j + 1) % n), (p + j, q + (j + 1) % n, q + j)]
            elif m > n:  # each vertex of the smaller ring closes four edges of the larger
                tris.append((q + (j + 1) % m, q + j, p + j // 4))
                if j % 4 == 3:
                    tris.append((q + (j + 1) % m, p + j // 4, p + (j // 4 + 1) % n))
            else:
                tris.append((p + j, p + (j + 1) % n, q + j // 4))
                if j % 4 == 3:
                    tris.append((p + (j + 1) % n, q + (j // 4 + 1) % m, q + j // 4))
    for first, n, flip in ((0, 6, True), (len(verts) - 6, 6, False)):
        for j in range(1, 5):
            t = (first, first + j, first + j + 1)
            tris.append(t[::-1] if flip else t)
    return np.array(verts) + [0.503, 0.498, 0.501], np.array(tris, np.int32)


def test_long_tube(ibm, orc):  # noqa: F811
    verts, tris = _tube(3, 100.0)
    _check(ibm, orc, verts, tris, (26, 27, 21), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def test_thin_faces_are_excluded(ibm):  # noqa: F811
    n, lo, hi = (96,) * 3, (0.0,) * 3, (1.0,) * 3
    fat, thin = (_seconds(ibm, *_tube(5, length), n, lo, hi) for length in (2.0, 8.0))
    print("sides above and below the angle of a thin face: %.0f us, %.0f us" % (1e6 * fat, 1e6 * thin))
    assert thin <= 4.0 * fat, (fat, thin)


@pytest.mark.parametrize("scale", [1e-3, 1e-5, 1e-9])
def test_small_bodies(ibm, orc, scale):  # noqa: F811
    verts, tris = W.uv_sphere(13, 18, 0.35 * scale, (0.503 * scale, 0.498 * scale, 0.501 * scale))
    _check(ibm, orc, verts, tris, (26, 27, 33), (0.0,) * 3, (scale,) * 3)


def test_small_bodies_are_searched_as_fast(ibm):  # noqa: F811
    n = (160,) * 3
    verts, tris = W.uv_sphere()
    plain = _seconds(ibm, verts, tris, n, (-2.0,) * 3, (2.0,) * 3)
    small = _seconds(ibm, verts * 1e-6, tris, n, (-2e-6,) * 3, (2e-6,) * 3)
    assert small <= 4.0 * plain, (plain, small)


def test_fine_meshes(ibm, orc):  # noqa: F811
    """Far more faces than cells: nodes with more than the hundred survivors that a warp keeps, thin faces among them."""
    verts, tris = W.uv_sphere(3, 4000, 0.35, (0.503, 0.498, 0.501))
    _check(ibm, orc, verts, tris, (14, 13, 12), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def test_fine_meshes_are_searched(ibm):  # noqa: F811
    """200,000 faces in three rings against 200,000 of usual shape: 700 times as long when a node of more survivors than a
    warp keeps evaluates every face, about 20 times as long when it evaluates the survivors."""
    n, lo, hi = (40,) * 3, (-2.0,) * 3, (2.0,) * 3
    plain, rings = (_seconds(ibm, *W.uv_sphere(a, b), n, lo, hi) for a, b in ((251, 400), (3, 50000)))
    print("usual shape %.0f us, three rings %.0f us" % (1e6 * plain, 1e6 * rings))
    assert rings <= 100.0 * plain, (plain, rings)
