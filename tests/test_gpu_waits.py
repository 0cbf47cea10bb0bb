"""The bounded waits of the kernels that wait for copies or neighbours within one launch: a copy that is never
started, or a CTA that never sends, ends the launch after the bound with the timeout flag set."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_10979_gb300 import flow, synth  # noqa: E402

KERNELS = {"tile": 0, "pdr": 1, "cluster": 2}


@pytest.mark.parametrize("kernel", list(KERNELS))
def test_a_wait_that_runs_out_is_reported_within_its_bound(kernel):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    k = KERNELS[kernel]
    to, parts = flow.of_wait_selftest(k, -1, 2000.0)
    assert to == 0 and parts > 1
    for withhold in (0, parts // 2, parts - 1):
        t0 = time.time()
        to, _ = flow.of_wait_selftest(k, withhold, 100.0)
        # a wait, the same again for the copies in flight, and at most one more for a neighbour's neighbours
        assert to == 1 and 0.1 <= time.time() - t0 < 2.0
    to, _ = flow.of_wait_selftest(k, -1, 2000.0)
    assert to == 0
    pr = synth.sinusoid_pair()
    ctx = flow.Context(0)
    st = flow.of_solve(ctx, torch.from_numpy(pr.I0).cuda(), torch.from_numpy(pr.I1).cuda(), flow.default_params())[3]
    assert st["energy"] == st["energy"]
    ctx.close()


def test_the_pairs_that_a_wait_leaves_unfinished_are_the_ones_reported():
    """A launch over three pairs whose last tile's copies never start: the last pair is reported, the others
    are finished; a block that gives up at its first tile reports the pairs of all its tiles."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    to, parts = flow.of_wait_selftest(3, -1, 2000.0)
    assert to == 0 and parts > 3 * 152
    assert flow.of_wait_selftest(3, parts - 1, 100.0)[0] == 4
    assert flow.of_wait_selftest(3, 0, 100.0)[0] & 1
    assert flow.of_wait_selftest(3, -1, 2000.0)[0] == 0
