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
