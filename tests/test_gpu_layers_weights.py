"""Layered blending with every pattern of zero weights: layers whose share is
zero are not sampled, the leading clips' among them (the first with a weight
then replaces what came before), and so is an additive layer of weight zero;
1 to 4 clips, with and without the layer, characters of different patterns
sharing an item, against the oracle (1e-4).  A clip that is off may hold
non-finite keys."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clips,additive", [(1, True), (2, False), (3, True), (4, False), (4, True)])
def test_zero_weight_patterns(clips, additive):
    rng = np.random.default_rng(clips * 2 + additive)
    chars = 96
    types = [synth.make_type(synth.relabel_dfs(synth.random_tree(n, d, rng, spine=d), rng)[0], rng, with_clips=True)
             for n, d in ((37, 9), (300, 25))]
    for t in types:
        t["keys"] = t["keys"][:min(clips, 2)]
    w = {"types": types, "char_type": (np.arange(chars) // 2 % 2).astype(np.int32),
         "time": rng.uniform(0, 0.2, chars).astype(np.float32), "weight": np.zeros(chars, np.float32)}
    w = synth.with_layers(w, n_clips=clips, additive=additive, seed=clips)
    on = (np.arange(chars)[:, None] >> np.arange(4)) & 1  # every pattern, all zeros among them
    w["weights"] = (rng.uniform(0.1, 1.0, (chars, 4)) * on).astype(np.float32)
    w["weights"][:, clips:] = 0
    w["add_w"][::3] = 0.0
    ctx, plan = _gpu.setup(w)
    args = [_gpu.cuda(w[k]) for k in ("time", "weights", "add_w")]
    got = ctx.evaluate_frame_layers(plan, *args)
    _gpu.assert_skin_close(got.cpu().numpy(), oracle.frame_layers(w), w)
    if clips == 4:  # the last clip off everywhere: its keys do not matter
        w["weights"][:, 3] = 0
        ref = oracle.frame_layers(w)
        for i, t in enumerate(types):
            keys = w["types"][i]["keys"].copy()
            keys[3] = np.nan
            ctx.upload_clips(i, keys, w["types"][i]["rate_hz"])
            if additive:
                ctx.upload_additive(i, w["types"][i]["add_keys"], w["types"][i]["rate_hz"])
        got = ctx.evaluate_frame_layers(plan, args[0], _gpu.cuda(w["weights"]), args[2])
        _gpu.assert_skin_close(got.cpu().numpy(), ref, w)
