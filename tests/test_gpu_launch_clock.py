"""dhq_last_launch_clock: the first CTA's run time and SM clock inside a launch of the observing instantiation."""
import pytest
import torch

import dhq_inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")


@pytest.mark.parametrize("width,n_linear,a_gran", [(64, 4, 0), (256, 4, 0), (256, 6, 1), (512, 4, 0), (512, 4, 1)])
def test_the_launch_clock_spans_the_launch(width, n_linear, a_gran):
    # weights that stay in shared memory (the copy warp is done at once) and weights that are streamed until the end
    dims = (2,) + (width,) * (n_linear - 1) + (3,)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 23)
    cd = to_dev(dhq_inputs.grid_coords(1024, 1024))
    out = torch.empty((cd.shape[0], 3), device="cuda")
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, a_gran=a_gran)
    try:
        dhq.dhq_calibrate(h, cd)
        for _ in range(3):
            dhq.dhq_forward_fused_debug(h, cd, out)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        dhq.dhq_forward_fused_debug(h, cd, out)
        t1.record()
        torch.cuda.synchronize()
        mhz, ms = dhq.dhq_last_launch_clock(h)
        # The events also see the launch itself and the CTA's setup (some 10 us of 120 us and more), and the first CTA may be done
        # one of its 27 rounds of tiles or more before the last.
        print(f"width {width}: {ms:.4f} ms in the kernel, {t0.elapsed_time(t1):.4f} ms between the events, {mhz:.0f} MHz")
        assert 0.75 * t0.elapsed_time(t1) <= ms <= 1.02 * t0.elapsed_time(t1)
        assert 500.0 < mhz < 2500.0
    finally:
        dhq.dhq_destroy(h)
