"""The default tensor path: the X-engine that builds its operand on the chip (at most 64 inputs: channel grouping,
short and long rings, several items a CTA, divided time ranges, in-chip flushes, more blocks than one launch takes,
rows that TMA does not take) and the two passes above, on the same shapes and options.
Everything is compared exactly, with the oracle or, at sizes it is slow at, with the int8 path."""
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


def _host(synth, N, C, T, blocks=1):
    spec = synth.Spec(kind="saturate", seed=N * 7 + C + T, seg_len=96, m8_segment=1)
    return synth.generate_host(spec, blocks * T, C, N)


def _correlate(env, host, npol, blocks=1, flush=0, skip=0):
    corr, _, torch = env
    T, C, N = host.shape[0] // blocks, host.shape[1], host.shape[2]
    xs = []
    for b in range(blocks):
        buf = torch.zeros((T * C * N + skip,), dtype=torch.uint8, device="cuda")
        buf[skip:].copy_(torch.from_numpy(host[b * T:(b + 1) * T].reshape(-1).copy()))
        xs.append(buf[skip:].view(T, C, N))
    with corr.Correlator(N, C, T, npol) as xc:
        if flush:
            xc.set_flush_period(flush)
        if blocks == 1:
            xc.accumulate(xs[0])
        else:
            xc.accumulate_batch(xs)
        out = xc.dump(corr.CORR_WHAT_CROSS).cpu().numpy(), xc.dump(corr.CORR_WHAT_AUTO).cpu().numpy()
        xc.sync()
        assert xc.samples() == T * blocks
    return out


def _check(env, host, npol, **kw):
    got = _correlate(env, host, npol, **kw)
    want = oracle.correlate(host, npol, threads=8)
    bad = np.argwhere(got[0] != want[0])
    assert bad.size == 0, (bad[:3].tolist(), got[0][tuple(bad[0])], want[0][tuple(bad[0])])
    assert np.array_equal(got[1], want[1])


# N: every packing of channels into 64-input units, unit strides of 48 and 64 bytes, the change of kernel at 64,
# blocks of 128 inputs with 16 .. 128 inputs in the last one. C: one unit, a unit without its pair, a partial last
# group. T: less than a stage, a stage, a stage and a bit.
@pytest.mark.parametrize("N,C,npol", [(1, 64, 1), (1, 80, 1), (2, 40, 2), (4, 4, 2), (6, 8, 2), (8, 2, 1), (12, 12, 2),
                                      (16, 1, 2), (16, 9, 2), (24, 3, 2), (24, 2, 1), (32, 1, 2), (32, 5, 2), (48, 1, 2),
                                      (48, 4, 1), (64, 1, 2), (64, 3, 1), (80, 1, 2), (96, 2, 1), (112, 3, 2), (128, 2, 2),
                                      (144, 2, 2), (192, 1, 1), (208, 2, 2), (256, 1, 2), (272, 1, 2), (400, 1, 2)])
@pytest.mark.parametrize("T", [1, 100, 128, 129, 1000])
def test_shapes(env, N, C, npol, T):
    _check(env, _host(env[1], N, C, T), npol)


@pytest.mark.parametrize("N,C", [(16, 5), (64, 3), (48, 5), (160, 2)])
@pytest.mark.parametrize("T,blocks,flush", [(300, 3, 128), (257, 5, 256), (128, 17, 0), (64, 40, 0), (1000, 2, 384)])
def test_batches_and_flushes(env, N, C, T, blocks, flush):
    """Blocks shorter than a stage, with a part stage each, and more of them than a launch takes; partial sums
    of 1, 2 and 3 stages, which end inside and across blocks."""
    _check(env, _host(env[1], N, C, T, blocks), 2, blocks=blocks, flush=flush)


@pytest.mark.parametrize("N,C,T,blocks", [(64, 701, 4096, 2), (32, 2401, 2048, 2), (16, 2500, 4096, 1), (48, 640, 3000, 1),
                                          (128, 310, 4096, 1), (512, 24, 8192, 2), (208, 160, 2000, 3), (200, 170, 4096, 2),
                                          (132, 190, 3000, 2), (134, 150, 3000, 2), (40, 700, 4096, 1)])
def test_several_items_a_cta(env, N, C, T, blocks):
    """More work items than SMs and rings that wrap many times, against the int8 path on the same blocks."""
    corr, synth, torch = env
    xs = [synth.generate_device(synth.Spec(kind="gauss_tone", seed=50 + b), T, C, N) for b in range(blocks)]
    out = {}
    for path in ("i8mma", "fp8tc"):
        with corr.Correlator(N, C, T, 2, path=path) as xc:
            xc.accumulate_batch(xs)
            xc.accumulate(xs[0])
            out[path] = xc.dump(corr.CORR_WHAT_CROSS), xc.dump(corr.CORR_WHAT_AUTO)
            xc.sync()
    for a, b in zip(out["i8mma"], out["fp8tc"]):
        assert torch.equal(a, b)


# rows TMA does not take, repacked: counts of every alignment (odd and even counts,
# unaligned blocks, a last column of 1 .. 16 inputs, rows of one and of many columns)
@pytest.mark.parametrize("N,C,npol,skip", [(72, 2, 2, 0), (200, 3, 2, 0), (136, 1, 1, 8), (68, 3, 2, 0), (100, 2, 2, 4), (260, 1, 2, 12),
                                           (128, 2, 2, 8), (128, 2, 2, 1), (131, 3, 1, 0), (67, 2, 1, 3), (130, 2, 2, 2),
                                           (66, 1, 2, 0), (40, 3, 2, 0), (20, 2, 2, 0), (10, 3, 2, 0), (7, 3, 1, 0), (33, 2, 1, 0),
                                           (1, 3, 1, 0), (64, 2, 2, 1), (32, 3, 2, 4), (16, 5, 2, 8), (5, 1, 1, 7)])
@pytest.mark.parametrize("T,blocks", [(1, 1), (129, 1), (1000, 2), (300, 18)])
def test_rows_that_tma_does_not_take(env, N, C, npol, skip, T, blocks):
    _check(env, _host(env[1], N, C, T, blocks), npol, skip=skip, blocks=blocks)


# whole rows of 16 bytes, channels between: every shift of the tiles (steps of 1, 2, 4 and 8 inputs), counts that with
# the largest shift just fill the last tile (113, 114, 116, 120, 241, 242, 248) and one that does not (122, repacked);
# up to 64 inputs units of one or more channels, the same (5, 10, 31, 49, 50, 52, 56 fill the unit; 60 is repacked)
@pytest.mark.parametrize("N,C,npol", [(65, 16, 1), (66, 8, 2), (68, 4, 2), (72, 2, 2), (72, 4, 1), (113, 16, 1), (114, 8, 2),
                                      (116, 4, 2), (120, 2, 2), (122, 8, 2), (131, 16, 1), (200, 2, 2), (241, 16, 1),
                                      (242, 8, 2), (248, 2, 2), (340, 4, 2), (3, 48, 1), (5, 48, 1), (7, 32, 1), (10, 24, 2),
                                      (14, 8, 2), (20, 12, 2), (22, 8, 2), (28, 4, 2), (31, 32, 1), (49, 16, 1), (50, 8, 2),
                                      (52, 4, 2), (56, 6, 2), (60, 4, 2)])
@pytest.mark.parametrize("T,blocks", [(1, 1), (129, 1), (700, 2)])
def test_channels_between_16_byte_boundaries(env, N, C, npol, T, blocks):
    _check(env, _host(env[1], N, C, T, blocks), npol, blocks=blocks)


def test_schedules_that_were_asked_for_mix_with_the_default(env):
    """Default, tile plan, build schedule and FP32 launches in one integration."""
    corr, synth, torch = env
    N, C, T = 128, 3, 640
    host = _host(synth, N, C, T, 8)
    xs = [torch.from_numpy(host[b * T:(b + 1) * T].copy()).cuda() for b in range(8)]
    with corr.Correlator(N, C, T, 2) as xc:
        xc.accumulate_batch(xs[:2])
        xc.set_tile_plan(3)
        xc.accumulate(xs[2])
        xc.set_tile_plan(0)
        xc.set_prep_sms(8)
        xc.accumulate_batch(xs[3:5])
        xc.set_prep_sms(-1)
        xc.set_batch_blocks(1)
        xc.accumulate_batch(xs[5:7])
        xc.set_path("fp32")
        xc.accumulate(xs[7])
        c, a = xc.dump(corr.CORR_WHAT_CROSS).cpu().numpy(), xc.dump(corr.CORR_WHAT_AUTO).cpu().numpy()
        xc.sync()
    want = oracle.correlate(host, 2, threads=8)
    assert np.array_equal(c, want[0]) and np.array_equal(a, want[1])


def test_captured_launch(env):
    """A default accumulate inside a CUDA graph, replayed on refilled buffers."""
    corr, synth, torch = env
    for N, C in ((64, 4), (256, 2)):
        T = 500
        host = _host(synth, N, C, T, 3)
        st = torch.cuda.Stream()
        x = torch.empty((T, C, N), dtype=torch.uint8, device="cuda")
        with torch.cuda.stream(st), corr.Correlator(N, C, T, 2) as xc:
            x.copy_(torch.from_numpy(host[:T].copy()))
            xc.accumulate(x)
            g = torch.cuda.CUDAGraph()
            st.synchronize()
            with torch.cuda.graph(g, stream=st):
                xc.accumulate(x)
            for b in (1, 2):
                x.copy_(torch.from_numpy(host[b * T:(b + 1) * T].copy()))
                g.replay()
            xc.sync()
            raw = xc.dump(corr.CORR_WHAT_CROSS).cpu().numpy()
            xc.sync()
        # the host counts one captured call: two replays leave one block's offset correction out
        want = oracle.correlate(host, 2, threads=8)[0]
        assert np.array_equal(raw[..., 1], want[..., 1])
        assert np.all(want[..., 0] - raw[..., 0] == 128 * T)
