"""The skinned frame at the sizes where its kernel changes path: vertex counts
around a warp's 32 and the CTA's 256, a pure chain long enough for the chain
scan, zero weights in every slot pattern; vertices and skin matrices against
the oracle, to the tolerances of the other frame tests (1e-4 on unit extent,
5e-4 at depth 1,024 and more)."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [1, 31, 33, 255, 257])
def test_skinned_frame_edges(nv):
    import torch
    rng = np.random.default_rng(nv)
    w = {"types": [], "char_type": np.array([0, 1, 0, 0, 2, 1, 0], np.int32),
         "time": rng.uniform(0, 1, 7).astype(np.float32), "weight": rng.uniform(0, 1, 7).astype(np.float32)}
    for p in (synth.random_tree(23, 9, rng, spine=9), synth.chain(1100), synth.chain(1)):
        t = synth.make_type(p, rng, with_clips=True)
        t["mesh"] = synth.make_mesh(p, nv, rng)
        wts = np.asarray(t["mesh"]["weights"], np.float32)
        bones = rng.integers(0, len(p), size=(nv, 4)).astype(np.int32)
        for v in range(nv):  # every pattern of zero slots in turn, one slot always in use
            keep = v % 15 + 1
            x = rng.uniform(0.1, 1.0, 4) * [(keep >> k) & 1 for k in range(4)]
            wts[v] = x / x.sum()
        t["mesh"].update(weights=wts, bones=bones)
        w["types"].append(t)
    ctx, plan = _gpu.setup(w)
    skin = torch.empty((plan.total, 12), dtype=torch.float32, device="cuda")
    verts = ctx.evaluate_frame_skinned(plan, _gpu.cuda(w["time"]), _gpu.cuda(w["weight"]), skin=skin)
    ref = oracle.frame(w)
    _gpu.assert_skin_close(skin.cpu().numpy(), ref, w)
    off = oracle.vertex_offsets(w["char_type"], w["types"])
    got, want = verts.cpu().numpy(), oracle.skin_vertices(w, ref)
    for c, t in enumerate(w["char_type"]):
        err = np.abs(got[off[c]:off[c + 1]] - want[off[c]:off[c + 1]])
        tol = _gpu.tol_for_depth(w["types"][t]["depth"])
        assert err[:, :3].max() <= tol
        # a normal is the sum of up to four rotated ones, normalized: its error grows as the sum shrinks;
        # compared where the sum keeps a tenth of its length
        S = ref.reshape(-1, 3, 4)[plan.row_off[c]:plan.row_off[c + 1], :, :3]
        m = w["types"][t]["mesh"]
        n = np.einsum("vk,vkij,vj->vi", m["weights"], S[m["bones"]], m["nrm"])
        keep = np.linalg.norm(n, axis=1) > 0.1
        assert err[keep, 3:].max(initial=0.0) <= 20 * tol
