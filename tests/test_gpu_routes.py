"""Calls that change the tensor path's route within one integration (the operand built on the chip, rows repacked into
the operand scratch first, the two passes over that scratch), and the total-power kernel for rows that TMA does not
take at the largest of its 16-bit sums. Whole numbers, exact."""
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


def _at(torch, host, skip):
    """A device copy of `host` that starts `skip` bytes into its buffer."""
    buf = torch.zeros(host.size + skip, dtype=torch.uint8, device="cuda")
    x = buf[skip:].view(host.shape)
    x.copy_(torch.from_numpy(host))
    return x


# at most 64 inputs built on the chip, in place and with the last unit partly filled; repacked rows; always two passes
@pytest.mark.parametrize("N,C", [(64, 3), (32, 5), (20, 4), (20, 3), (31, 2), (63, 1), (128, 3), (72, 2)])
def test_routes_mix_in_one_integration(env, N, C):
    """Default, tile plans, build schedules, batches and unaligned blocks, with the operand scratch kept throughout:
    what one route leaves there does not reach another's sums."""
    corr, synth, torch = env
    T, npol, n = 300, 1 if N % 2 else 2, 14
    host = synth.generate_host(synth.Spec(kind="gauss_tone", seed=N + C), n * T, C, N)
    xs = [_at(torch, host[b * T:(b + 1) * T], 1 if b in (3, 9) else 0) for b in range(n)]
    with corr.Correlator(N, C, T, npol) as xc:
        xc.accumulate_batch(xs[:2])
        xc.set_tile_plan(1)
        xc.accumulate(xs[2])
        xc.set_tile_plan(0)
        xc.accumulate(xs[3])
        xc.set_tile_plan(3)
        xc.accumulate_batch(xs[4:6])
        xc.set_tile_plan(2)
        xc.accumulate(xs[6])
        xc.set_tile_plan(0)
        xc.accumulate_batch(xs[7:9])
        xc.set_prep_sms(8)
        xc.accumulate(xs[9])
        xc.accumulate_batch(xs[10:12])
        xc.set_prep_sms(-1)
        xc.accumulate_batch(xs[12:])
        cross, autos = xc.dump(corr.CORR_WHAT_CROSS).cpu().numpy(), xc.dump(corr.CORR_WHAT_AUTO).cpu().numpy()
        xc.sync()
    want = oracle.correlate(host, npol, threads=8)
    assert np.array_equal(cross, want[0]) and np.array_equal(autos, want[1])


@pytest.mark.parametrize("unaligned", [(0,), (1,), (0, 1, 2, 3), (4,)])
def test_batch_whose_blocks_take_different_routes(env, unaligned):
    """64 inputs x 3 channels: aligned blocks are read in place, the others repacked; a mixed batch takes the two
    passes."""
    corr, synth, torch = env
    N, C, T, n = 64, 3, 200, 5
    host = synth.generate_host(synth.Spec(kind="gauss_tone", seed=9), n * T, C, N)
    xs = [_at(torch, host[b * T:(b + 1) * T], 3 if b in unaligned else 0) for b in range(n)]
    with corr.Correlator(N, C, T, 2) as xc:
        xc.accumulate_batch(xs)
        cross, autos = xc.dump(corr.CORR_WHAT_CROSS).cpu().numpy(), xc.dump(corr.CORR_WHAT_AUTO).cpu().numpy()
        xc.sync()
    want = oracle.correlate(host, 2, threads=8)
    assert np.array_equal(cross, want[0]) and np.array_equal(autos, want[1])


def test_total_power_of_the_largest_samples_in_rows_of_any_alignment(env):
    """-8 - 8 i throughout in a buffer that starts at an odd address, so that TMA does not take its rows: 1400 blocks of
    columns fill the GPU, so a block takes the most rows it may, 504 a warp, and every 16-bit sum reaches
    504 x 128 = 64512; then one column, and the rows left over."""
    corr, _, torch = env
    for N, C, T in ((1024, 700, 4500), (17, 1, 20000)):
        x = torch.full((T * C * N + 1,), 0x88, dtype=torch.uint8, device="cuda")[1:].view(T, C, N)
        with corr.Correlator(N, C, T, 1 if N % 2 else 2) as xc:
            xc.accumulate_autos(x)
            assert torch.all(xc.dump(corr.CORR_WHAT_AUTO) == 128 * T).item()
            xc.sync()
