"""The batch schedule knobs and their autotuner: every launch length gives the oracle's sums, and
corr_autotune leaves zeroed accumulators, a valid schedule that then correlates bit-exactly, and a
cached choice for the next context of the same shape."""
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


def _blocks(env, N, C, T, n, seed):
    _, synth, torch = env
    host = synth.generate_host(synth.Spec(kind="gauss_tone", seed=seed), n * T, C, N)
    return host, [torch.from_numpy(np.ascontiguousarray(host[b * T:(b + 1) * T])).cuda() for b in range(n)]


def test_every_launch_length_matches_the_oracle(env):
    corr, _, torch = env
    N, C, T, npol, n = 144, 3, 1000, 2, 7
    host, blocks = _blocks(env, N, C, T, n, 41)
    want_c, want_a = oracle.correlate(host, npol, threads=8)
    with corr.Correlator(N, C, T, npol) as xc:
        default = xc.batch_blocks
        assert default == corr.corr_batch_blocks(N, C, T, npol)
        for K in (1, 2, 3, 7, 0):
            xc.set_batch_blocks(K)
            assert xc.batch_blocks == (K or default)
            xc.accumulate_batch(blocks)
            c = xc.dump(corr.CORR_WHAT_CROSS, reset=True).cpu().numpy()
            a = xc.dump(corr.CORR_WHAT_AUTO, reset=True).cpu().numpy()
            xc.sync()
            assert np.array_equal(c, want_c) and np.array_equal(a, want_a), K
        for bad in (-1, 1 << 20):
            with pytest.raises(corr.CorrError):
                xc.set_batch_blocks(bad)


def test_autotune_then_correlate(env):
    corr, _, torch = env
    N, C, T, npol, n = 256, 3, 4096, 2, 12
    host, blocks = _blocks(env, N, C, T, n, 43)
    want_c, want_a = oracle.correlate(host, npol, threads=8)
    with corr.Correlator(N, C, T, npol) as xc:
        choice = xc.autotune(blocks, reps=1)
        assert choice["tile_plan"] in (0, 1, 2, 3) and choice["batch_blocks"] >= 1 and choice["n_tried"] >= 6
        assert choice["ms_per_block"] > 0
        assert (xc.tile_plan, xc.batch_blocks, xc.prep_sms) == (choice["tile_plan"], choice["batch_blocks"],
                                                                choice["prep_sms"])
        assert xc.samples(corr.CORR_WHAT_CROSS) == 0 and xc.samples(corr.CORR_WHAT_AUTO) == 0
        assert not torch.any(xc.dump(corr.CORR_WHAT_CROSS) != 0).item()
        xc.accumulate_batch(blocks)
        c = xc.dump(corr.CORR_WHAT_CROSS).cpu().numpy()
        a = xc.dump(corr.CORR_WHAT_AUTO).cpu().numpy()
        xc.sync()
    assert np.array_equal(c, want_c) and np.array_equal(a, want_a)
    # the same shape again: the cached choice, applied without timing
    with corr.Correlator(N, C, T, npol) as xc:
        again = xc.autotune(blocks, reps=1)
        assert again["n_tried"] == 0
        assert (again["tile_plan"], again["batch_blocks"], again["prep_sms"]) == (
            choice["tile_plan"], choice["batch_blocks"], choice["prep_sms"])


def test_autotune_needs_the_tensor_path(env):
    corr, _, torch = env
    _, blocks = _blocks(env, 64, 1, 256, 2, 5)
    with corr.Correlator(64, 1, 256, 2, path="fp32") as xc:
        with pytest.raises(corr.CorrError):
            xc.autotune(blocks)


# run in a process of its own: the tuner reads the file named by CORR_AUTOTUNE_CACHE once
TUNE = """
import sys, torch
sys.path.insert(0, %r)
from paper_1411_3751_gb300 import corr
for n in (64, 256):
    blocks = [torch.zeros((128, 2, n), dtype=torch.uint8, device="cuda") for _ in range(3)]
    with corr.Correlator(n, 2, 128, 2) as xc:
        c = xc.autotune(blocks, reps=1)
        print("tuned", n, c["n_tried"] > 0, c["tile_plan"], c["batch_blocks"], c["prep_sms"])
"""


def test_saved_schedules_of_small_arrays_from_earlier_versions_are_timed_anew(env, tmp_path):
    """A "batch" line holds for more than 64 inputs; at most 64 have a tag of their own, since what was saved for them
    before would keep them in the two passes."""
    import os
    import subprocess
    import sys

    _, _, torch = env
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cache = tmp_path / "tuned"
    line = "%%s %%d 2 128 2 %d 3 1 2 0 0.001000" % sms

    def tune():
        r = subprocess.run([sys.executable, "-c", TUNE % root], capture_output=True, text=True, timeout=300,
                           env=dict(os.environ, CORR_AUTOTUNE_CACHE=str(cache)))
        assert r.returncode == 0, r.stderr[-2000:]
        return [t.split()[1:] for t in r.stdout.splitlines() if t.startswith("tuned")]

    cache.write_text(line % ("batch", 64) + "\n" + line % ("batch", 256) + "\n")
    small, large = tune()
    assert small[:2] == ["64", "True"] and large == ["256", "False", "1", "2", "0"]
    assert [t.split()[:2] for t in cache.read_text().splitlines()[2:]] == [["batch64", "64"]]
    cache.write_text(line % ("batch64", 64) + "\n" + line % ("batch64", 256) + "\n")
    small, large = tune()
    assert small == ["64", "False", "1", "2", "0"] and large[:2] == ["256", "True"]


@pytest.mark.parametrize("plan,blocks,prep", [(9, 2, 0), (-1, 2, 0), (1, 0, 0), (1, 20000000, 0), (1, 2, 100000), (1, 2, -5)])
def test_impossible_saved_schedules_are_not_applied(env, tmp_path, plan, blocks, prep):
    """A damaged line (no such tile plan, no or more blocks a launch than the operand buffer may hold, no such number of
    SMs) is timed anew: 20 million blocks a launch of this shape would overflow the sample offsets."""
    import os
    import subprocess
    import sys

    _, _, torch = env
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cache = tmp_path / "tuned"
    cache.write_text("batch 256 2 128 2 %d 3 %d %d %d 0.001000\n" % (sms, plan, blocks, prep))
    r = subprocess.run([sys.executable, "-c", TUNE % root], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CORR_AUTOTUNE_CACHE=str(cache)))
    assert r.returncode == 0, r.stderr[-2000:]
    assert any(t.split()[1:3] == ["256", "True"] for t in r.stdout.splitlines() if t.startswith("tuned"))
