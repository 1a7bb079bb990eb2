"""3-D pre-processing at the sizes where its word- and cluster-wise forms change path, bit for bit against the FP64
oracle: lattice rows around the 32-node word, a body that leaves the lattice, one-node axes, a mesh of a few large
faces and one whose pole joins more faces than a node keeps, flat faces that the FP32 bounds may not judge, and
coordinates far from the origin."""
import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W
from test_gpu_geometry3d import _check, ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(31, 12, 13), (32, 12, 13), (33, 12, 13), (64, 9, 10), (65, 9, 10), (95, 8, 8),
                               (12, 40, 7), (7, 12, 70)])
def test_rows_around_the_word(ibm, orc, n):  # noqa: F811
    verts, tris = W.uv_sphere(9, 12, 0.31, (0.52, 0.47, 0.49))
    _check(ibm, orc, verts, tris, n, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


@pytest.mark.parametrize("n,lo,hi", [
    ((40, 36, 33), (0.3, 0.1, 0.45), (1.1, 0.6, 1.3)),       # the body leaves the lattice on four sides
    ((1, 30, 30), (0.4, 0.0, 0.0), (0.6, 1.0, 1.0)),         # one node along an axis
    ((30, 1, 1), (0.0, 0.4, 0.4), (1.0, 0.6, 0.6)),
    ((20, 20, 20), (2.0, 2.0, 2.0), (3.0, 3.0, 3.0)),        # no node in the bounding box
])
def test_lattice_against_the_box(ibm, orc, n, lo, hi):  # noqa: F811
    verts, tris = W.uv_sphere(11, 16, 0.35, (0.5, 0.5, 0.5))
    _check(ibm, orc, verts, tris, n, lo, hi)


def test_few_large_faces(ibm, orc):  # noqa: F811
    verts, tris = W.box_mesh((-0.41, -0.33, -0.27), (0.43, 0.36, 0.29))
    _check(ibm, orc, verts, tris, (70, 33, 41), (-1.0, -1.0, -1.0), (1.0, 1.0, 1.0))


def test_pole_of_many_faces(ibm, orc):  # noqa: F811
    """Nodes near the poles lie closest to a vertex of 150 faces: more survivors than a node keeps."""
    verts, tris = W.uv_sphere(6, 150, 0.4, (0.501, 0.499, 0.5))
    _check(ibm, orc, verts, tris, (21, 21, 40), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def test_flat_faces_and_two_bodies(ibm, orc):  # noqa: F811
    """A long thin box (faces of extreme aspect ratio) beside a sphere, as one surface of two closed parts."""
    v0, t0 = W.box_mesh((0.1, 0.2, 0.2), (0.9, 0.20002, 0.4))
    v1, t1 = W.uv_sphere(7, 10, 0.2, (0.5, 0.65, 0.55))
    _check(ibm, orc, np.concatenate([v0, v1]), np.concatenate([t0, t1 + len(v0)]).astype(np.int32), (33, 41, 29),
           (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def test_far_from_the_origin(ibm, orc):  # noqa: F811
    verts, tris = W.uv_sphere(13, 18, 0.35, (1000.5, -2000.5, 300.5))
    _check(ibm, orc, verts, tris, (30, 31, 33), (1000.0, -2001.0, 300.0), (1001.0, -2000.0, 301.0))
