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


def test_total_power_of_the_largest_samples(env):
    """-8 - 8 i throughout: 128 a sample, every 16-bit sum of a full run of rows at its largest."""
    corr, synth, torch = env
    for N, C, T in ((1024, 700, 4500), (16, 1, 20000)):
        x = torch.full((T, C, N), 0x88, dtype=torch.uint8, device="cuda")
        with corr.Correlator(N, C, T, 2) as xc:
            xc.accumulate_autos(x)
            assert torch.all(xc.dump(corr.CORR_WHAT_AUTO) == 128 * T).item()
            xc.sync()


# channels of one block, of several blocks and of a block and a bit; both polarisation counts
@pytest.mark.parametrize("N,C,T,npol", [(2, 5, 77, 2), (1, 3, 50, 1), (64, 7, 301, 2), (91, 3, 301, 1), (130, 2, 999, 2),
                                        (260, 2, 129, 2)])
@pytest.mark.parametrize("skip", [0, 1])
def test_dump_restarts_and_alignments(env, N, C, T, npol, skip):
    corr, synth, torch = env
    host = synth.generate_host(synth.Spec(kind="saturate", seed=N + T, seg_len=64, m8_segment=1), 2 * T, C, N)
    x = [torch.from_numpy(host[i * T:(i + 1) * T].copy()).cuda() for i in range(2)]
    with corr.Correlator(N, C, T, npol) as xc:
        for what, k in ((corr.CORR_WHAT_CROSS, 0), (corr.CORR_WHAT_AUTO, 1)):
            for fmt, f in ((corr.CORR_FMT_CI64, oracle.FMT_CI64), (corr.CORR_FMT_CF32, oracle.FMT_CF32),
                           (corr.CORR_FMT_CF32_NORM, oracle.FMT_CF32_NORM)):
                dtype = torch.int64 if fmt == corr.CORR_FMT_CI64 else torch.float32
                for block in (0, 1):  # each dump restarts: the second holds the second block alone
                    xc.accumulate(x[block])
                    out = _at_offset(torch, xc.out_shape(what), dtype, skip)
                    xc.dump(what, fmt, reset=True, out=out)
                    want = oracle.correlate(host[block * T:(block + 1) * T], npol)[k]
                    assert np.array_equal(out.cpu().numpy(), oracle.to_format(want, f, T)), (what, fmt, block)
                    assert xc.samples(what) == 0
                xc.reset()
        xc.sync()


def test_normalised_dump_is_the_nearest_float(env):
    """70 million quotients of sums by an odd count, all near 2^24 distinct numerators: the FP64-free
    division and its fallback near ties against the double division."""
    corr, synth, torch = env
    N, C, T = 512, 64, 8001
    x = synth.generate_device(synth.Spec(kind="gauss_tone", seed=8), T, C, N)
    with corr.Correlator(N, C, T, 2) as xc:
        xc.accumulate(x)
        v = xc.dump(corr.CORR_WHAT_CROSS)
        q = xc.dump(corr.CORR_WHAT_CROSS, corr.CORR_FMT_CF32_NORM)
        assert torch.equal(q, (v.double() / float(T)).float())
        xc.sync()


# sums about 2^30, 2^31 and past 32 bits (one input pair of the most negative samples, a few of them different), both signs
@pytest.mark.parametrize("T", [(1 << 23) + 5, (1 << 24) - 1, (1 << 24) + 9, (1 << 25) + 3])
@pytest.mark.parametrize("npol", [1, 2])
def test_normalised_dump_of_large_sums(env, T, npol):
    corr, _, torch = env
    x = torch.full((T, 1, 4), 0x88, dtype=torch.uint8, device="cuda")
    x[:, 0, 2] = 0x78  # 7 - 8i: products of both signs in both parts
    x[::1001, 0, 1] = 0x3F
    with corr.Correlator(4, 1, T, npol) as xc:
        xc.accumulate(x)
        v = xc.dump(corr.CORR_WHAT_CROSS)
        assert int(v.abs().max()) > 1 << 30
        q = xc.dump(corr.CORR_WHAT_CROSS, corr.CORR_FMT_CF32_NORM)
        f = xc.dump(corr.CORR_WHAT_CROSS, corr.CORR_FMT_CF32)
        xc.sync()
    assert torch.equal(q, (v.double() / float(T)).float())
    assert torch.equal(f, v.float())


# a few columns, many columns, a last partial column, one sample, a split time range; odd pointers
@pytest.mark.parametrize("N,C,T", [(1, 1, 1), (2, 3, 5000), (7, 5, 65), (512, 3, 63), (33, 31, 129), (256, 400, 40),
                                   (3, 1, 9001), (512, 160, 4100)])
# and runs of the rows at the most that 16-bit sums hold, of the largest samples
@pytest.mark.parametrize("skip", [0, 1, 5])
def test_total_power_columns(env, N, C, T, skip):
    corr, synth, torch = env
    host = synth.generate_host(synth.Spec(kind="saturate", seed=N * 3 + T, seg_len=32, m8_segment=0), T, C, N)
    x = _at_offset(torch, host.shape, torch.uint8, skip)
    x.copy_(torch.from_numpy(host))
    with corr.Correlator(N, C, T, 1) as xc:
        xc.accumulate_autos(x)
        xc.accumulate_autos(x)
        a = xc.dump(corr.CORR_WHAT_AUTO)
        xc.sync()
    assert np.array_equal(a.cpu().numpy(), 2 * oracle.autos(host))


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


# chunks of 64 channels: one, an edge, a last one of 1; rows divided into segments of one and of several chunks, with
# a shorter last one; more rows than are divided
@pytest.mark.parametrize("N,T,F,chan0,C", [(1, 1, 64, 0, 64), (33, 1, 200, 1, 65), (40, 2, 4096, 0, 4096), (35, 3, 700, 9, 641),
                                           (512, 40, 1100, 3, 1090), (512, 300, 140, 0, 129), (30, 6000, 70, 2, 66)])
def test_requantize_segments(env, N, T, F, chan0, C):
    corr, _, torch = env
    x = np.random.default_rng(N + T).integers(-1 << 17, 1 << 17, (N, T, F, 2), dtype=np.int32)
    got = corr.requantize(torch.from_numpy(x).cuda(), chan0, C, gain=2.0 ** -14).cpu().numpy()
    assert np.array_equal(got, oracle.requantize(x, chan0, C, gain=2.0 ** -14))


# every tap count that has its own kernel, and the loop beyond them; one and an odd number of spectra
@pytest.mark.parametrize("n_taps", [1, 2, 3, 4, 5, 6, 7, 8, 9, 17])
@pytest.mark.parametrize("n_spectra", [1, 5])
def test_pfb_tap_counts(env, n_taps, n_spectra):
    """Within 4 log2(8192) FP32 roundings of each spectrum's L2 norm of the float64 oracle, as in the filterbank's tests."""
    corr, _, torch = env
    M = 8192
    adc = np.random.default_rng(n_taps).integers(-128, 128, (3, (n_spectra + n_taps - 1) * M), dtype=np.int8)
    X = corr.pfb(torch.from_numpy(adc).cuda(), n_taps=n_taps).cpu().numpy()
    want, y = oracle.pfb(adc, M, n_taps), oracle.pfb_fir(adc, M, n_taps)
    tol = 4 * 13 * 2.0 ** -24 * 2.0 ** -13 * np.sqrt(M) * np.sqrt((y.astype(np.float64) ** 2).sum(-1))
    assert np.all(np.abs(X[..., 0] + 1j * X[..., 1] - want).max(axis=-1) <= tol)
