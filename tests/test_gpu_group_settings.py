"""Groups whose members' settings change between calls: a captured launch reads only what the group owns, or is
refused, against the oracle."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1411_3751_gb300 import corr, synth

    assert torch.cuda.is_available()
    return corr, synth, torch


def _blocks(synth, shapes, T, k):
    return [synth.generate_device(synth.Spec(kind="gauss_tone", seed=60 + i), T, c, n, t0=k * T)
            for i, (n, c) in enumerate(shapes)]


def _check(corr, g, blocks, npol):
    for i, m in enumerate(g.members):
        cross, autos = m.dump(corr.CORR_WHAT_CROSS), m.dump(corr.CORR_WHAT_AUTO)
        m.sync()
        want = oracle.correlate(np.concatenate([b[i].cpu().numpy() for b in blocks]), npol, threads=8)
        assert np.array_equal(cross.cpu().numpy(), want[0]) and np.array_equal(autos.cpu().numpy(), want[1]), i


@pytest.mark.parametrize("shapes", [[(200, 6), (64, 4), (512, 3)], [(66, 9), (130, 2), (20, 3)]])
def test_captured_group_outlives_its_members_work_lists(env, shapes):
    """A member's tile plan is set anew after the capture, which frees its work list, and the freed memory is written:
    the replayed launch correlates as it was captured."""
    corr, synth, torch = env
    T, npol = 600, 2
    blk = [_blocks(synth, shapes, T, k) for k in range(2)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), corr.Group(shapes, T, npol) as g:
        bufs = [torch.empty_like(b) for b in blk[0]]
        g.capture(bufs, stream)
        for plan in (1, 2, 3, 0):
            for m in g.members:
                m.set_tile_plan(plan)
        with corr.Correlator(512, 64, 128, npol) as other:  # its lists and buffers may take the freed memory
            other.set_tile_plan(1)
            for k in range(2):
                for dst, src in zip(bufs, blk[k]):
                    dst.copy_(src)
                g.launch(stream)
            _check(corr, g, blk, npol)


@pytest.mark.parametrize("release", ["path", "batch_blocks"])
def test_captured_group_is_refused_once_its_scratch_is_gone(env, release):
    """A member's operand scratch is released after the capture (by its path, by its blocks per launch): the graph that
    writes there is not launched, and a new capture works. Members that do not go through the scratch do not matter."""
    corr, synth, torch = env
    shapes, T, npol = [(64, 4), (200, 3)], 600, 2
    blk = _blocks(synth, shapes, T, 0)

    def let_go(m):
        if release == "path":
            m.set_path("fp32")
            m.set_path("fp8tc")
        else:
            m.set_batch_blocks(1 if m.batch_blocks > 1 else 2)

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), corr.Group(shapes, T, npol) as g:
        stream.synchronize()
        g.capture(blk, stream)
        let_go(g.members[0])  # 64 inputs: correlated without the scratch
        g.launch(stream)
        let_go(g.members[1])
        with pytest.raises(corr.CorrError):
            g.launch(stream)
        _check(corr, g, [blk], npol)  # the refused launch was not counted
        g.capture(blk, stream)
        g.launch(stream)
        _check(corr, g, [blk, blk], npol)


@pytest.mark.parametrize("shapes,T", [([(256, 4)] * 8, 700), ([(66, 5), (68, 3), (131, 2), (72, 4), (512, 2), (128, 3), (65, 1), (67, 7)], 1001),
                                      ([(130, 3), (20, 4), (130, 3)], 130), ([(512, 1), (64, 2)], 300)])
def test_members_that_share_a_launch(env, shapes, T):
    """Groups whose larger members share one build and one X-engine launch: equal and uneven members, rows of every load
    width, members without a share in it between them, a single larger member; two blocks, then a replayed graph."""
    corr, synth, torch = env
    npol = 1 if any(n % 2 for n, _ in shapes) else 2
    blk = [_blocks(synth, shapes, T, k) for k in range(3)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), corr.Group(shapes, T, npol) as g:
        g.accumulate(blk[0])
        g.accumulate(blk[1])
        g.capture(blk[2], stream)
        g.launch(stream)
        _check(corr, g, blk, npol)


def test_members_on_sm_pairs_beside_a_shared_launch(env):
    """Blocks of more than 5632 samples and enough items for the 512-input member to launch by itself on SM pairs,
    beside two members that share a launch and one on the 64-input kernel: every cell against the int8 path."""
    corr, synth, torch = env
    shapes, T, npol = [(512, 64), (128, 9), (64, 5), (200, 6)], 5700, 2
    blk = _blocks(synth, shapes, T, 0)
    with corr.Group(shapes, T, npol) as g:
        g.accumulate(blk)
        for (n, c), m, b in zip(shapes, g.members, blk):
            with corr.Correlator(n, c, T, npol, path="i8mma") as ref:
                ref.accumulate(b)
                for what in (corr.CORR_WHAT_CROSS, corr.CORR_WHAT_AUTO):
                    assert torch.equal(m.dump(what), ref.dump(what)), (n, what)
            m.sync()


# run in a process of its own: the tuner reads the file named by CORR_AUTOTUNE_CACHE once
TUNE = """
import sys, torch
sys.path.insert(0, %r)
from paper_1411_3751_gb300 import corr, synth
shapes, T = %r, %d
blk = [synth.generate_device(synth.Spec(kind="gauss_tone", seed=i), T, c, n) for i, (n, c) in enumerate(shapes)]
with corr.Group(shapes, T, 2) as g:
    g.members[0].set_tile_plan(1)
    plans = g.autotune(blk)
    assert plans == [m.tile_plan for m in g.members]
    g.accumulate(blk)
    for m, (n, c), b in zip(g.members, shapes, blk):
        with corr.Correlator(n, c, T, 2, path="i8mma") as ref:
            ref.accumulate(b)
            assert torch.equal(m.dump(corr.CORR_WHAT_CROSS), ref.dump(corr.CORR_WHAT_CROSS))
    g.members[0].sync()
print("plans", plans)
"""


def test_group_autotuner_chooses_among_what_the_group_runs(env, tmp_path):
    """Members without a tile plan keep the default; the 512-input member that launches by itself on SM pairs can stay
    there. Plans that an earlier version saved for members of the same shapes are not applied; the new ones are."""
    import os
    import re
    import subprocess
    import sys

    corr, _, torch = env
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shapes, T = [(64, 4), (32, 5), (512, 64), (200, 3)], 5700
    cache = tmp_path / "tuned"

    def tune(lines):
        cache.write_text("".join(line + "\n" for line in lines))
        r = subprocess.run([sys.executable, "-c", TUNE % (root, shapes, T)], capture_output=True, text=True, timeout=300,
                           env=dict(os.environ, CORR_AUTOTUNE_CACHE=str(cache)))
        assert r.returncode == 0, r.stderr[-2000:]
        saved = cache.read_text().splitlines()[len(lines):]
        return [int(p) for p in re.search(r"plans \[(.*)\]", r.stdout).group(1).split(",")], saved

    old = ["%d %d %d 2 %d 1" % (n, c, T, sms) for n, c in shapes]
    plans, saved = tune(old)
    assert plans[:2] == [0, 0] and plans[2] in (0, 1, 3) and plans[3] in (0, 1)
    # timed and saved anew: the two members that have a choice, nothing for the others
    assert [line.split()[:3] for line in saved] == [["group", "512", "64"], ["group", "200", "3"]]
    for want in (3, 1):  # a saved choice among the plans that the launch can run is applied without timing
        plans, again = tune(["group 512 64 %d 2 %d 1 %d" % (T, sms, want), "group 200 3 %d 2 %d 0 1" % (T, sms)])
        assert plans == [0, 0, want, 1] and not again
