"""Raster of meshes with more vertices than a character's stage in shared
memory (4,096), alone and beside staged ones in one plan: every kind of
triangle of test_gpu_raster.py (slivers, sizes on both sides of 64 pixels,
positions past the 32-bit range, vertices only 4-byte aligned); and of
triangles from 64 pixels to the whole image, wide, tall and square, among
small ones; id for id against the oracle under that file's rule for equal
depths."""
import numpy as np
import pytest

import oracle
from .test_gpu_raster import _mesh

pytestmark = pytest.mark.gpu


def _depths(idents, at, meshes, verts, types, cols, spacing, ox, oy, scale):
    """Depths of triangles `idents` at the pixel centre `at`, in float64."""
    out = []
    for i in idents:
        c, f = int(i) >> 12, int(i) & 4095
        v = verts[c][meshes[types[c]][1][f]].astype(np.float64)
        x, y = ox + scale * (v[:, 0] + c % cols * spacing), oy - scale * (v[:, 1] - c // cols * spacing)
        lam = np.linalg.solve(np.stack([x, y, np.ones(3)]), [at[1] + 0.5, at[0] + 0.5, 1.0])
        out.append(float(lam @ ((2.0 - v[:, 2]) / 4.0)))
    return out


@pytest.mark.parametrize("kind,sizes,nf,shift", [
    ("strip", [4097], 4095, 0), ("slivers", [4500], 257, 1), ("large", [5000], 40, 0), ("far", [4200], 64, 3),
    ("random", [6000, 60], 500, 0), ("slivers", [90, 4097, 4096], 300, 3)])
def test_meshes_past_the_stage(kind, sizes, nf, shift):
    rng = np.random.default_rng(sum(sizes) + nf)
    _check([_mesh(kind, nv, nf, rng) for nv in sizes], 160, 96, 8.0, shift)


@pytest.mark.parametrize("wide,high,width,height", [(70, 3, 997, 40), (3, 70, 37, 641), (64, 64, 320, 200),
                                                    (300, 200, 640, 360), (900, 9, 997, 33), (5, 600, 31, 641)])
def test_triangles_of_many_pixels(wide, high, width, height):
    rng = np.random.default_rng(wide * 7 + high)
    pos = np.zeros((90, 3), np.float32)  # 64 pixels per unit: positions are whole quarter pixels
    pos[:, 0] = rng.integers(-2 * wide, 2 * wide + 1, 90) / 256.0
    pos[:, 1] = rng.integers(-2 * high, 2 * high + 1, 90) / 256.0
    pos[60:, :2] /= 16.0
    pos[:, 2] = np.arange(90) * 0.6180339887 % 1.0
    faces = np.concatenate([rng.integers(0, 60, (45, 3)), rng.integers(60, 90, (30, 3))]).astype(np.int32)
    _check([(pos, rng.permutation(faces))], width, height, 64.0, 0)


def _check(meshes, width, height, scale, shift):
    import torch
    import paper_2505_06703_gb300 as pk
    sizes = [len(m[0]) for m in meshes]
    n = len(sizes)
    types = np.arange(7) % n
    verts = []
    for c, t in enumerate(types):
        v = np.zeros((sizes[t], 6), np.float32)
        v[:, :3] = meshes[t][0]
        v[:, 2] += c * 0.0137
        v[:, 5] = 1.0
        verts.append(v)
    flat = np.concatenate(verts)
    ctx = pk.Context(0)
    ids = ctx.create_skeletons([np.array([-1], np.int32)] * n, rest_q=[np.array([[0, 0, 0, 1]], np.float32)] * n,
                               rest_t=[np.zeros((1, 3), np.float32)] * n)
    for i, nv, (pos, faces) in zip(ids, sizes, meshes):
        ctx.upload_mesh(i, {"pos": pos, "nrm": np.tile(np.array([[0, 0, 1]], np.float32), (nv, 1)),
                            "bones": np.zeros((nv, 4), np.int32),
                            "weights": np.tile(np.array([[1, 0, 0, 0]], np.float32), (nv, 1))})
        ctx.upload_faces(i, faces)
    plan = ctx.plan(np.asarray(ids, np.int32)[types])
    buf = torch.zeros(flat.size + 8, device="cuda")
    dev = buf[shift:shift + flat.size].view(-1, 6)
    dev.copy_(torch.as_tensor(flat))
    view = (3, 32.0 / scale, 12.0, 10.0, scale)
    got, _ = ctx.raster(plan, dev, width, height, *view)
    got = got.cpu().numpy().view(np.uint32)
    off = np.concatenate([[0], np.cumsum([sizes[t] for t in types])])
    ref = oracle.raster([meshes[t][1] for t in types], flat.astype(np.float64), off, *view, width, height)
    empty = oracle.RASTER_EMPTY
    assert (ref != empty).any() and np.array_equal(got == empty, ref == empty)
    for at in np.argwhere(got != ref):
        d = _depths((got[tuple(at)], ref[tuple(at)]), at, meshes, verts, types, *view)
        assert abs(d[0] - d[1]) < 4e-7, (at, d)
