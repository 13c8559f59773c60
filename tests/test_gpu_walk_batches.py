"""The chain-walk kernel takes a frame's walkable types from a batch size on
(165 joints per step squared of the longest schedule), the segmented kernel
below: batches on both sides of that line, for schedules of different lane
counts and chunk lengths (a bush of 32 lanes, trees, short chains) and one or
two clips, against the oracle to the frame tests' tolerance."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu

BUSH = np.array([-1] + [0] * 63 + list(range(1, 64)), np.int32)  # 63 chains of two joints off the root, interleaved


@pytest.mark.parametrize("walk", [1, 2])
@pytest.mark.parametrize("shape,chars", [("chain6", 40), ("chain6", 2000), ("tree24", 300), ("tree24", 1500),
                                         ("bush", 100), ("bush", 900), ("tree67", 200), ("tree67", 1500),
                                         ("mixed", 60), ("mixed", 1800)])
def test_walk_batches(shape, chars, walk):
    rng = np.random.default_rng(chars + walk)
    tree = lambda n, d: synth.relabel_dfs(synth.random_tree(n, d, rng, spine=d), rng)[0]
    parents = {"chain6": lambda: [synth.chain(6)], "tree24": lambda: [tree(24, 8)],
               "bush": lambda: [synth.relabel_dfs(BUSH, rng)[0]], "tree67": lambda: [tree(67, 14)],
               "mixed": lambda: [tree(24, 8), tree(67, 14), synth.chain(600)]}[shape]()
    types = [synth.make_type(p, rng, with_clips=True) for p in parents]
    types[0]["keys"] = types[0]["keys"][:1 + chars % 3]  # one clip where chars is a multiple of 3
    ct = (np.arange(chars) % len(types)).astype(np.int32)
    ct[ct == 2] = np.where(rng.uniform(size=(ct == 2).sum()) < 0.02, 2, 1)
    w = {"types": types, "char_type": ct, "time": rng.uniform(-1, 2, chars).astype(np.float32),
         "weight": rng.uniform(0, 1, chars).astype(np.float32)}
    ctx, plan = _gpu.setup(w)
    ctx.set_schedule(plan, [16, 2, 2048, walk, 0])
    for _ in range(2):
        out = ctx.evaluate_frame(plan, _gpu.cuda(w["time"]), _gpu.cuda(w["weight"]))
    _gpu.assert_skin_close(out.cpu().numpy(), oracle.frame(w), w)
    assert ctx.status() == 0
