"""Work-item sizes follow the batch (items shrink until they fill the resident
CTAs): batches just below and above one and two waves of 304 CTAs, mixed with
a type whose characters are too long to share an item; plain frame on the
segmented kernel, forward and backward against the oracle, to the tolerances
of the other tests (gradients 5e-4 of their largest: depth 1,300)."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chars", [1, 152, 303, 305, 607, 913])
def test_batches_around_whole_waves(chars):
    rng = np.random.default_rng(chars)
    types = [synth.make_type(synth.relabel_dfs(synth.random_tree(n, d, rng, spine=d), rng)[0], rng, with_clips=True)
             for n, d in ((19, 7), (61, 20))] + [synth.make_type(synth.chain(1300), rng, with_clips=True)]
    ct = rng.integers(0, 2, chars).astype(np.int32)
    ct[::200] = 2
    rows = int(sum(len(types[t]["parents"]) for t in ct))
    w = {"types": types, "char_type": ct, "time": rng.uniform(0, 1, chars).astype(np.float32),
         "weight": rng.uniform(0, 1, chars).astype(np.float32)}
    w["q"], w["t"] = synth.local_poses(rng, rows, unnormalized=True, t_scale=min(t["scale"] for t in types))
    g = rng.uniform(-1, 1, size=(rows, 3)).astype(np.float32)
    ctx, plan = _gpu.setup(w)
    q, t = _gpu.cuda(w["q"]), _gpu.cuda(w["t"])
    ctx.set_schedule(plan, [16, 2, 2048, 0, 0])
    _gpu.assert_skin_close(ctx.evaluate_frame(plan, _gpu.cuda(w["time"]), _gpu.cuda(w["weight"])).cpu().numpy(),
                           oracle.frame(w), w)
    skin, _ = ctx.forward_local(plan, q, t)
    _gpu.assert_skin_close(skin.cpu().numpy(), oracle.forward_qt(types, ct, w["q"], w["t"])[0], w)
    dq, dt = oracle.grad(types, ct, w["q"], w["t"], g.astype(np.float64))
    scale = max(1.0, np.abs(dq).max(), np.abs(dt).max())
    for adj in (0, 6):
        ctx.set_schedule(plan, [16, 2, 2048, 0, adj])
        gq, gt = ctx.backward(plan, q, t, _gpu.cuda(g))
        assert np.abs(gq.cpu().numpy() - dq).max() <= 5e-4 * scale
        assert np.abs(gt.cpu().numpy() - dt).max() <= 5e-4 * scale
