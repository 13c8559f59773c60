"""The host-buffer frame cuts a plan of at least 1,024 characters into up to four
ranges of growing joint counts, none shorter than its frame takes to copy:
batches of one, two and four ranges against the oracle, to the frame tests'
tolerance."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("joints,chars", [(3, 1024), (3, 1500), (40, 1200), (40, 2500), (40, 4100)])
def test_host_frame_ranges(joints, chars):
    import torch
    rng = np.random.default_rng(joints + chars)
    tree = synth.relabel_dfs(synth.random_tree(joints, min(joints, 9), rng, spine=min(joints, 9)), rng)[0]
    types = [synth.make_type(p, rng, with_clips=True) for p in (tree, synth.chain(5))]
    w = {"types": types, "char_type": (np.arange(chars) % 7 == 0).astype(np.int32),
         "time": rng.uniform(-1, 2, chars).astype(np.float32), "weight": rng.uniform(0, 1, chars).astype(np.float32)}
    ctx, plan = _gpu.setup(w)
    ref = oracle.frame(w)
    host = [torch.as_tensor(w[k]).pin_memory() for k in ("time", "weight")]
    for _ in range(2):
        out = ctx.evaluate_frame_host(plan, *host)
        torch.cuda.synchronize()
        _gpu.assert_skin_close(out.numpy(), ref, w)
    assert ctx.status() == 0
