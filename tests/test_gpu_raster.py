"""The raster kernel's paths against the oracle's rasterizer, id for id.

Vertices lie on a grid that float32 and float64 snap alike (multiples of 1/64
times powers of two), so both sides decide coverage from the same integers:
the images must be equal, except where the two answers' depths agree to 4e-7,
what float32 rounding of both (three products below 0.5, a sum, the reciprocal
area) can turn around.  The cases are the
sizes where the kernel changes its path: triangles around 64 pixels (32-bit
edge functions below, 64-bit from there), positions past the 32-bit range,
meshes past the staged vertex count, vertices that are only 4-byte aligned,
characters wholly or partly outside the image, face counts around the 32
triangles a warp sets up at once, slivers along rows, columns and diagonals.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _mesh(kind, nv, nf, rng):
    """(positions [nv, 3] in model units, faces): screen pixels are 8 per unit below."""
    z = (np.arange(nv) * 0.6180339887 % 1.0)[:, None]  # depths apart
    if kind == "slivers":
        base = rng.integers(-128, 128, size=(nv, 2)) / 64.0
        pos = base.copy()
        pos[1::3] = base[0::3][:len(pos[1::3])] + rng.integers(-2, 3, size=pos[1::3].shape) / 64.0
        along = rng.integers(0, 3, size=nv)
        pos[along == 1, 0] = 0.5
        pos[along == 2, 1] = -0.25
    elif kind == "large":  # 40 to 90 pixels across: both sides of the 64-pixel line
        pos = rng.integers(-360, 360, size=(nv, 2)) / 64.0
    elif kind == "far":  # a third of the corners far past the 32-bit range
        pos = rng.integers(-256, 256, size=(nv, 2)) / 64.0
        pos[::7, 0] *= 2.0 ** 18
        pos[3::7, 1] *= 2.0 ** 18
    else:
        pos = rng.integers(-128, 128, size=(nv, 2)) / 64.0
    faces = rng.integers(0, nv, size=(nf, 3)) if kind != "strip" else (np.arange(nf)[:, None] + np.arange(3)) % nv
    return np.concatenate([pos, z], axis=1).astype(np.float32), faces.astype(np.int32)


def _depth(ident, px, py, verts, faces, cols, spacing, ox, oy, scale):
    """Depth of triangle `ident` at a pixel centre, in float64."""
    c, f = int(ident) >> 12, int(ident) & 4095
    v = verts[c, faces[f]].astype(np.float64)
    x, y = ox + scale * (v[:, 0] + c % cols * spacing), oy - scale * (v[:, 1] - c // cols * spacing)
    lam = np.linalg.solve(np.stack([x, y, np.ones(3)]), [px + 0.5, py + 0.5, 1.0])
    return float(lam @ ((2.0 - v[:, 2]) / 4.0))


@pytest.mark.parametrize("kind,nv,nf,chars,width,height,shift", [
    ("strip", 3, 1, 3, 64, 48, 0),
    ("strip", 1500, 1498, 12, 160, 96, 0),
    ("slivers", 301, 257, 9, 97, 61, 0),
    ("slivers", 300, 31, 9, 97, 61, 1),
    ("slivers", 300, 33, 9, 96, 64, 3),
    ("large", 64, 40, 6, 320, 200, 0),
    ("far", 90, 64, 6, 160, 120, 0),
    ("random", 4096, 500, 4, 128, 96, 0),
    ("random", 4097, 500, 4, 128, 96, 0),
    ("random", 50, 40, 40, 1, 1, 0),
    ("random", 50, 4096, 4, 33, 7, 0),
])
def test_raster_paths_equal_oracle(kind, nv, nf, chars, width, height, shift):
    import torch
    import paper_2505_06703_gb300 as pk
    rng = np.random.default_rng(nv * 31 + nf + width)
    pos, faces = _mesh(kind, nv, nf, rng)
    verts = np.zeros((chars, nv, 6), np.float32)
    verts[..., :3] = pos
    verts[..., 2] += (np.arange(chars) * 0.0137)[:, None]
    verts[..., 5] = 1.0
    ctx = pk.Context(0)
    ids = ctx.create_skeletons([np.array([-1], np.int32)], rest_q=[np.array([[0, 0, 0, 1]], np.float32)],
                               rest_t=[np.zeros((1, 3), np.float32)])
    ctx.upload_mesh(ids[0], {"pos": pos, "nrm": np.tile(np.array([[0, 0, 1]], np.float32), (nv, 1)),
                             "bones": np.zeros((nv, 4), np.int32),
                             "weights": np.tile(np.array([[1, 0, 0, 0]], np.float32), (nv, 1))})
    ctx.upload_faces(ids[0], faces)
    plan = ctx.plan(np.zeros(chars, np.int32))
    buf = torch.zeros(verts.size + 8, device="cuda")
    dev = buf[shift:shift + verts.size].view(-1, 6)
    dev.copy_(torch.as_tensor(verts.reshape(-1, 6)))
    cols, spacing, ox, oy, scale = 3, 4.0, 12.0, 10.0, 8.0
    got, _ = ctx.raster(plan, dev, width, height, cols, spacing, ox, oy, scale)
    ref = oracle.raster([faces] * chars, verts.reshape(-1, 6).astype(np.float64), np.arange(chars + 1) * nv, cols,
                        spacing, ox, oy, scale, width, height)
    got = got.cpu().numpy().view(np.uint32)
    empty = oracle.RASTER_EMPTY
    assert np.array_equal(got == empty, ref == empty)
    at = (verts, faces, cols, spacing, ox, oy, scale)
    for py, px in np.argwhere(got != ref):
        d = [_depth(i, px, py, *at) for i in (got[py, px], ref[py, px])]
        assert abs(d[0] - d[1]) < 4e-7, (py, px, got[py, px], ref[py, px], d)
    assert (kind, width) == ("random", 1) or (ref != oracle.RASTER_EMPTY).any()
