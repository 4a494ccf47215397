"""The batched form's tuner: an engine without trajectories in the sample keeps its configuration, a small
sample tunes the kernels that large runs take, and what it sets holds for later runs."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300.simulator import BatchSimulator  # noqa: E402


def test_only_engines_in_the_sample_are_tuned():
    n = 24
    traj, noise = list(range(n)), [dict(W.STRESS)] * n
    with BatchSimulator(2, "cr", max_traj=4096) as b:
        before = b.config()
        warps, ms = b.autotune(5, traj, ["c128u", "c64u"] * (n // 2), noise)
        assert warps == before[0] == b.config()[0] and ms > 0
        b.set_config(10, 3, 128)
        warps, ms = b.autotune(5, traj, ["c128", "c64"] * (n // 2), noise)
        assert b.config()[1:] == (3, 128) and b.config()[0] == warps and ms > 0


def test_small_sample_does_not_settle_on_a_shape_that_starves_large_runs():
    # warps that an SM holds by warps per CTA: 10, 8, 6, 8, 10 for 2, 4, 6, 8, 10 (22 KiB each): 6 is a tenth slower
    n = 32
    with BatchSimulator(2, "cr", max_traj=8192) as b:
        for seed in range(4):
            warps, _ = b.autotune(seed, list(range(n)), ["c128"] * n, [dict(W.STRESS)] * n)
            assert warps != 6


def test_a_refused_configuration_leaves_no_trace():
    from paper_2204_11404_gb300 import capi

    n = 8
    args = (5, list(range(n)), ["c128", "c64", "c128u", "c64u"] * 2, [dict(W.STRESS)] * n)
    with BatchSimulator(2, "cr", max_traj=16) as b:
        ref = b.run(*args)
        for bad in ((0, 4, 256), (-3, 4, 256), (11, 4, 256), (64, 4, 256), (8, 1, 256), (8, 7, 256), (8, 4, 100)):
            before = b.config()
            with pytest.raises(capi.QecError):
                b.set_config(*bad)
            assert b.config()[1:] == before[1:]
            for x, y in zip(b.run(*args), ref):      # the refusal is not reported again by the next run
                assert (x == y).all()
