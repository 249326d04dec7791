"""The memory-bound kernels at the sizes where they can go wrong: dumps (unit and channel edges, outputs at
odd alignments, the fused restart), the total-power kernel (ragged columns, unaligned buffers, split
time ranges) and the corner turn's granules. Whole numbers and bytes are compared exactly; normalised
values are the float nearest to the double quotient, so they are compared exactly too."""
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


def _at_offset(torch, shape, dtype, skip):
    """A contiguous tensor of `shape` that starts `skip` elements into its buffer."""
    n = int(np.prod(shape))
    return torch.full((n + skip,), 7, dtype=dtype, device="cuda")[skip:].view(shape)


# granules of 16, 8, 4, 2 and 1 bytes; empty parts; runs longer than a piece; more columns than a block
@pytest.mark.parametrize("T,C,n_local,chan_b,in_b", [
    (3, 300, 32, [0, 109, 109, 300], [0, 16, 48]), (2, 40, 24, [0, 0, 40], [0, 8, 24, 24]), (5, 7, 12, [0, 3, 7], [0, 4, 20]),
    (4, 9, 10, [0, 9], [0, 10, 26]), (2, 1500, 7, [0, 1499, 1500], [0, 301, 601]), (17, 5, 16, [0, 2, 5], [0, 4096, 8192])])
@pytest.mark.parametrize("skip", [0, 4])
def test_corner_turn_granules(env, T, C, n_local, chan_b, in_b, skip):
    corr, _, torch = env
    st = torch.cuda.current_stream().cuda_stream
    g = np.random.default_rng(T * C)
    x = g.integers(0, 256, (T, C, n_local), dtype=np.uint8)
    d_in, d_out = _at_offset(torch, x.shape, torch.uint8, skip), _at_offset(torch, (x.size,), torch.uint8, skip)
    d_in.copy_(torch.from_numpy(x))
    corr.corr_corner_turn_pack(d_in.data_ptr(), T, C, n_local, chan_b, d_out.data_ptr(), st)
    want = np.concatenate([x[:, a:b].ravel() for a, b in zip(chan_b, chan_b[1:])])
    assert np.array_equal(d_out.cpu().numpy(), want)
    N = in_b[-1]
    y = g.integers(0, 256, (T, C, N), dtype=np.uint8)
    src = np.concatenate([y[:, :, a:b].ravel() for a, b in zip(in_b, in_b[1:])])
    d_in, d_out = _at_offset(torch, src.shape, torch.uint8, skip), _at_offset(torch, y.shape, torch.uint8, skip)
    d_in.copy_(torch.from_numpy(src))
    corr.corr_corner_turn_unpack(d_in.data_ptr(), T, C, N, in_b, d_out.data_ptr(), st)
    assert np.array_equal(d_out.cpu().numpy(), y)
