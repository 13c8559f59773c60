"""The prefix over the segment tree (pass 2 of the scan) on tree shapes that
exercise its tables: no links, one link, link counts around powers of two,
forests whose segments need different numbers of steps, stars, combs and
random topological orders, at several segment lengths and batch sizes;
forward (model and skin) and adjoint against the oracle, to the tolerances of
the other tests (1e-4 on unit extent; gradients 1e-4 of their largest)."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu


def _comb(teeth):
    """A spine numbered so that every joint is its own segment: joint 2k + 1 hangs off joint 2k as a leaf and the
    spine goes on from joint 2k, so joint 2k has k links."""
    par = [-1]
    for k in range(teeth):
        par += [2 * k, 2 * k]
    return np.array(par, np.int32)


def _forest(rng):
    par = []
    for teeth in (0, 1, 2, 3, 5, 8, 9, 17):
        base = len(par)
        par += [p if p < 0 else p + base for p in _comb(teeth)]
    return np.array(par, np.int32)


SHAPES = {
    "one": lambda rng: np.array([-1], np.int32),
    "star": lambda rng: np.array([-1] + [0] * 40, np.int32),
    "comb2": lambda rng: _comb(2), "comb3": lambda rng: _comb(3), "comb4": lambda rng: _comb(4),
    "comb5": lambda rng: _comb(5), "comb64": lambda rng: _comb(64), "comb65": lambda rng: _comb(65),
    "forest": _forest,
    "chain": lambda rng: synth.chain(300),
    "topological": lambda rng: synth.relabel_random_topological(synth.random_tree(150, 40, rng, spine=40), rng)[0],
    "tree": lambda rng: synth.relabel_dfs(synth.random_tree(331, 60, rng, spine=60), rng)[0],
}


@pytest.mark.parametrize("seg_len", [1, 4, 16])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_segment_prefix_shapes(shape, seg_len):
    rng = np.random.default_rng(len(shape) * 7 + seg_len)
    typ = synth.make_type(SHAPES[shape](rng), rng, with_clips=False)
    n = len(typ["parents"])
    for chars in (1, 7, 70):
        w = {"types": [typ], "char_type": np.zeros(chars, np.int32)}
        w["q"], w["t"] = synth.local_poses(rng, chars * n, unnormalized=True, t_scale=typ["scale"])
        g = rng.uniform(-1, 1, size=(chars * n, 3)).astype(np.float32)
        ctx, plan = _gpu.setup(w, with_clips=False)
        for adj in (0, 4):
            ctx.set_schedule(plan, [seg_len, 2, 2048, 1, adj])
            q, t = _gpu.cuda(w["q"]), _gpu.cuda(w["t"])
            skin, model = ctx.forward_local(plan, q, t, model=True)
            S, M = oracle.forward_qt(w["types"], w["char_type"], w["q"], w["t"])
            assert np.abs(skin.cpu().numpy().reshape(-1, 3, 4) - S).max() <= 1e-4
            assert np.abs(model.cpu().numpy().reshape(-1, 3, 4) - M).max() <= 1e-4
            gq, gt = ctx.backward(plan, q, t, _gpu.cuda(g))
            dq, dt = oracle.grad(w["types"], w["char_type"], w["q"], w["t"], g.astype(np.float64))
            scale = max(1.0, np.abs(dq).max(), np.abs(dt).max())
            assert np.abs(gq.cpu().numpy() - dq).max() <= 1e-4 * scale
            assert np.abs(gt.cpu().numpy() - dt).max() <= 1e-4 * scale
