"""Skinned vertices without a weight to share: all four zero, or subnormal
ones that cannot be halved.  Their zero slots are skipped like any other's, so
the non-finite pose of a bone that only they name does not reach the vertex."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu

TINY = float(np.float32(1.4e-45))  # the smallest subnormal


def test_vertices_without_weight():
    rng = np.random.default_rng(3)
    n, chars = 6, 40
    t = synth.make_type(synth.chain(n), rng, with_clips=True)
    # joint 5's position overflows; 0 to 4 stay finite.  The same in every key
    t["keys"] = t["keys"].copy()
    t["keys"][..., :4] = [0, 0, 0, 1]
    t["keys"][..., 4, 4] = 3e38
    t["keys"][..., 5, 4] = 3e38
    t["rest_q"] = np.tile(np.array([0, 0, 0, 1], np.float32), (n, 1))
    w4 = np.array([[0, 0, 0, 0], [-0.0, 0, 0, 0], [0, TINY, 0, 0], [0, 0, 3 * TINY, TINY], [1, 0, 0, 0],
                   [0, 0, 0, 1], [0.5, 0, 0.5, 0], [TINY, 0, 0, 0]] * 12, np.float32)
    bones = np.where(w4 == 0, 5, rng.integers(0, 4, size=w4.shape)).astype(np.int32)
    nv = len(w4)
    nrm = np.tile(np.array([[0, 0, 1]], np.float32), (nv, 1))
    t["mesh"] = {"pos": rng.uniform(-0.5, 0.5, (nv, 3)).astype(np.float32), "nrm": nrm, "bones": bones,
                 "weights": w4, "faces": np.zeros((0, 3), np.int32)}
    w = {"types": [t], "char_type": np.zeros(chars, np.int32), "time": rng.uniform(0, 1, chars).astype(np.float32),
         "weight": rng.uniform(0, 1, chars).astype(np.float32)}
    ctx, plan = _gpu.setup(w)
    import torch
    skin = torch.empty((plan.total, 12), device="cuda")
    got = ctx.evaluate_frame_skinned(plan, _gpu.cuda(w["time"]), _gpu.cuda(w["weight"]), skin=skin).cpu().numpy()
    S = skin.cpu().numpy().reshape(chars, n, 3, 4)
    assert not np.isfinite(S[:, 5]).all() and np.isfinite(S[:, :4]).all()
    got = got.reshape(chars, nv, 6)
    assert np.isfinite(got).all()
    none = (w4 == 0).all(axis=1)
    assert (got[:, none] == 0).all()
    used = w4.astype(np.float64)[None, :, :, None]
    rows = np.where(used[..., None] != 0, S.astype(np.float64)[:, np.minimum(bones, 4)], 0.0)  # unused slots out
    p1 = np.concatenate([t["mesh"]["pos"], np.ones((nv, 1))], axis=1).astype(np.float64)
    want = (used * np.einsum("cvkij,vj->cvki", rows, p1)).sum(axis=2)
    assert np.abs(got[..., :3] - want).max() <= 1e-5  # four products of values below 2, in float32
    full = w4.max(axis=1) == 1
    assert np.abs(got[:, full, 3:] - [0, 0, 1]).max() <= 1e-5
