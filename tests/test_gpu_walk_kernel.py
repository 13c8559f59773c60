"""The chain-walk kernels on batches of every size: a schedule whose fourth
value is 1 runs every walkable type on the walk, with three warps per item or,
with one clip and few items or past 8.5 item slots per SM, with one; anim_plan_walk says which.  Frames back to back and in a graph, key counts
on both sides of the work queue's 32, inverse binds from every source, every
lane count from 1 to 32 (chunks of 4, 2 and 1 steps), forests and joints not
numbered depth first, against the oracle to the frame tests' tolerance."""
import numpy as np
import pytest

import oracle
import synth
from . import _gpu

pytestmark = pytest.mark.gpu

WALK = [16, 2, 2048, 1, 0]


def _comb(chains, length):
    """A root with `chains` chains of `length` joints, numbered chain by chain: one lane per chain."""
    par = [-1]
    for _ in range(chains):
        par += [0] + list(range(len(par), len(par) + length - 1))
    return np.array(par, np.int32)


def _workload(parents, chars, rng, clips=2):
    types = [synth.make_type(p, rng, with_clips=True) for p in parents]
    for t in types:
        t["keys"] = t["keys"][:clips]
    return {"types": types, "char_type": (np.arange(chars) % len(types)).astype(np.int32),
            "time": rng.uniform(-1, 2, chars).astype(np.float32), "weight": rng.uniform(0, 1, chars).astype(np.float32)}


def _inputs(w):
    return _gpu.cuda(w["time"]), _gpu.cuda(w["weight"])


def _joints(w, types):
    return sum(len(w["types"][t]["parents"]) for t in w["char_type"] if t in types)


@pytest.mark.parametrize("parents,lanes", [
    (synth.chain(6), 1), (synth.chain(160), 1), (_comb(2, 12), 2), (_comb(4, 20), 4), (_comb(8, 30), 8),
    (_comb(16, 20), 16), (_comb(32, 10), 32), (np.array([-1] + [0] * 599, np.int32), 32),
    (np.array([-1] + [0] * 63 + list(range(1, 64)), np.int32), 32), (np.array([-1, 0, -1, 2, 2, -1], np.int32), 2)])
@pytest.mark.parametrize("clips", [1, 2])
def test_lane_counts(parents, lanes, clips):
    rng = np.random.default_rng(len(parents) + clips)
    for chars in (1, 33, 130):
        w = _workload([parents], chars, rng, clips)
        ctx, plan = _gpu.setup(w)
        ctx.set_schedule(plan, WALK)
        assert ctx.plan_walk(plan) == (plan.total, lanes, 1 if clips == 1 else 3)
        out = ctx.evaluate_frame(plan, *_inputs(w))
        _gpu.assert_skin_close(out.cpu().numpy(), oracle.frame(w), w)
        ctx.set_schedule(plan, [16, 2, 2048, 0, 0])
        assert ctx.plan_walk(plan) == (0, 0, 0)


@pytest.mark.parametrize("parents,lanes,chars,warps", [
    (_comb(32, 10), 32, 1100, 3), (_comb(32, 10), 32, 1400, 1), (_comb(32, 10), 32, 2700, 1),
    (_comb(16, 20), 16, 2300, 3), (_comb(16, 20), 16, 3000, 1), (_comb(4, 4), 4, 8000, 3), (_comb(4, 4), 4, 12000, 1)])
def test_warps_by_items(parents, lanes, chars, warps):
    """Two clips: one warp per item past 8.5 item slots (of 152 SMs) per SM."""
    rng = np.random.default_rng(chars)
    w = _workload([parents], chars, rng)
    ctx, plan = _gpu.setup(w)
    ctx.set_schedule(plan, WALK)
    assert ctx.plan_walk(plan) == (plan.total, lanes, warps)
    out = ctx.evaluate_frame(plan, *_inputs(w))
    _gpu.assert_skin_close(out.cpu().numpy(), oracle.frame(w), w)
    assert ctx.status() == 0


def test_many_characters_beside_many_branch_points():
    """A type of 32 characters per item beside one of some 170 branch-point slots per character: each item takes the
    slots its own type needs (the largest of both at once would not fit a CTA)."""
    rng = np.random.default_rng(3)
    tree = synth.relabel_dfs(synth.random_tree(1000, 40, rng, spine=40), rng)[0]
    w = _workload([synth.chain(6), tree, _comb(8, 30)], 90, rng)
    ctx, plan = _gpu.setup(w)
    ctx.set_schedule(plan, WALK)
    assert ctx.plan_walk(plan)[0] == plan.total
    out = ctx.evaluate_frame(plan, *_inputs(w))
    _gpu.assert_skin_close(out.cpu().numpy(), oracle.frame(w), w)
    assert ctx.status() == 0


@pytest.mark.parametrize("dragons", [0, 1, 40])  # none, chained on the stream, side by side
@pytest.mark.parametrize("clips", [1, 2])
def test_frames_in_a_row_and_in_a_graph(dragons, clips):
    import torch
    rng = np.random.default_rng(dragons * 2 + clips)
    tree = synth.relabel_random_topological(synth.random_tree(67, 14, rng, spine=14), rng)[0]
    w = _workload([tree, synth.chain(40)], 500, rng, clips)
    w["types"].append(synth.make_type(synth.chain(600), rng, with_clips=True))
    w["char_type"][:dragons] = 2
    frames = [dict(w, time=rng.uniform(0, 1, 500).astype(np.float32), weight=rng.uniform(0, 1, 500).astype(np.float32))
              for _ in range(6)]
    ref = [oracle.frame(f) for f in frames]
    ctx, plan = _gpu.setup(w)
    ctx.set_schedule(plan, WALK)
    assert ctx.plan_walk(plan)[::2] == (_joints(w, (0, 1)), 1 if clips == 1 else 3)
    ins = [_inputs(f) for f in frames]
    outs = [torch.zeros((plan.total, 12), device="cuda") for _ in frames]
    torch.cuda.synchronize()
    for (tm, wt), o in zip(ins, outs):
        ctx.evaluate_frame(plan, tm, wt, out=o)
    for o, r in zip(outs, ref):
        _gpu.assert_skin_close(o.cpu().numpy(), r, w)
    # two frames per graph, replayed on inputs that change in place
    eager = [o.clone() for o in outs]
    bufs = [(torch.zeros(500, device="cuda"), torch.zeros(500, device="cuda")) for _ in range(2)]
    pair = outs[:2]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for (tm, wt), o in zip(bufs, pair):
            ctx.evaluate_frame(plan, tm, wt, out=o)
    for k in (0, 2, 4):
        for i in range(2):
            for dst, src in zip(bufs[i], ins[k + i]):
                dst.copy_(src)
        g.replay()
        for i in range(2):
            assert torch.equal(pair[i], eager[k + i]), (k, i)
    assert ctx.status() == 0


@pytest.mark.parametrize("keys", [2, 3, 32, 33, 40])
@pytest.mark.parametrize("clips", [1, 2])
def test_key_counts(keys, clips):
    rng = np.random.default_rng(keys + 100 * clips)
    w = _workload([synth.random_tree(48, 9, rng, spine=9), synth.chain(64)], 400, rng, clips)
    for t in w["types"]:
        k = t["keys"]
        t["keys"] = np.ascontiguousarray(np.concatenate([k] * -(-keys // k.shape[1]), axis=1)[:, :keys])
    ctx, plan = _gpu.setup(w)
    ctx.set_schedule(plan, WALK)
    assert ctx.plan_walk(plan)[0] == plan.total
    out = ctx.evaluate_frame(plan, *_inputs(w))
    _gpu.assert_skin_close(out.cpu().numpy(), oracle.frame(w), w)
    assert ctx.status() == 0


@pytest.mark.parametrize("bind", ["rigid", "scaled"])
def test_given_inverse_binds(bind):
    import paper_2505_06703_gb300 as pk
    rng = np.random.default_rng(7)
    w = _workload([synth.random_tree(96, 20, rng, spine=20), synth.chain(30)], 100, rng)
    Bs = [oracle.inverse_bind(t["parents"], t["rest_q"], t["rest_t"]).astype(np.float32) for t in w["types"]]
    scale = 1.5 if bind == "scaled" else 1.0
    for B in Bs:
        B[:, :, :3] *= scale
    _, M = oracle.frame(w, want_model=True)
    ref = oracle.bind(M, np.concatenate([Bs[t] for t in w["char_type"]]).astype(np.float64))
    ctx = pk.Context(0)
    ids = ctx.create_skeletons([t["parents"] for t in w["types"]], inv_bind=Bs)
    for i, t in zip(ids, w["types"]):
        ctx.upload_clips(i, t["keys"], t["rate_hz"])
    plan = ctx.plan(np.asarray(ids, np.int32)[w["char_type"]])
    ctx.set_schedule(plan, WALK)
    assert ctx.plan_walk(plan)[0] == (plan.total if bind == "rigid" else 0)  # a scaled bind is never walked
    out = ctx.evaluate_frame(plan, *_inputs(w))
    for ty, e in _gpu.per_type_maxabs(out.cpu().numpy(), ref, w).items():
        assert e <= scale * _gpu.tol_for_depth(w["types"][ty]["depth"]), (ty, e)


@pytest.mark.parametrize("small,props,walked", [(6200, 2, (0,)), (6200, 400, ()), (3000, 2, ()), (6200, 0, (0,))])
def test_rare_long_type_beside_a_crowd(small, props, walked):
    """By batch: a 67-joint crowd large enough for the walk keeps it beside a few 150-joint chains, whose own line
    lies at millions of joints; not beside chains that are a seventh of the joints, nor below 400 thousand."""
    rng = np.random.default_rng(small + props)
    tree = synth.relabel_dfs(synth.random_tree(67, 14, rng, spine=14), rng)[0]
    w = _workload([tree, synth.chain(150)], small + props, rng)
    w["char_type"][:] = 0
    w["char_type"][rng.permutation(small + props)[:props]] = 1
    ctx, plan = _gpu.setup(w)
    assert ctx.get_schedule(plan)[3] == 2
    assert ctx.plan_walk(plan)[0] == _joints(w, walked)
    out = ctx.evaluate_frame(plan, *_inputs(w))
    _gpu.assert_skin_close(out.cpu().numpy(), oracle.frame(w), w)
    ctx.set_schedule(plan, [16, 2, 2048, 1, 0])
    assert ctx.plan_walk(plan)[0] == plan.total


@pytest.mark.parametrize("chars,dragons", [(1500, 0), (4000, 3)])
def test_host_frame_runs_on_the_device_frames_kernels(chars, dragons):
    """The ranges of a host-buffer frame are below the walk's line where the whole batch is above it: they follow the
    whole batch, so both entry points give the same bits."""
    import torch
    rng = np.random.default_rng(chars)
    tree = synth.relabel_dfs(synth.random_tree(67, 14, rng, spine=14), rng)[0]
    w = _workload([tree, synth.chain(600)], chars, rng)
    w["char_type"][:] = 0
    w["char_type"][rng.permutation(chars)[:dragons]] = 1
    ctx, plan = _gpu.setup(w)
    assert ctx.plan_walk(plan)[0] == 67 * (chars - dragons)
    ref = ctx.evaluate_frame(plan, *_inputs(w)).cpu()
    host = [torch.as_tensor(w[k]).pin_memory() for k in ("time", "weight")]
    for _ in range(2):
        out = ctx.evaluate_frame_host(plan, *host)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    ctx.set_schedule(plan, [16, 2, 2048, 0, 0])  # the ranges follow a new schedule too
    ref = ctx.evaluate_frame(plan, *_inputs(w)).cpu()
    out = ctx.evaluate_frame_host(plan, *host)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
