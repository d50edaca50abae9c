"""Launches of at most one tile per SM take kernels of their own (all epilogue warps on one tile; up to 64
tokens per SM tiles of 64): on either side of these borders and at ragged ends dhq_forward must return the bits of the observed fused
kernel, whose per-layer values the other tests compare with the definition."""
import numpy as np
import pytest
import torch

import dhq_inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")

KINDS = [dict(), dict(w_gran=1, a_gran=1), dict(rotation=2), dict(rotation=2, a_gran=1), dict(w_bits=4, a_bits=4, w_gran=1, a_gran=1),
         dict(rotation=1), dict(rotation=1, a_gran=1), dict(activation=1, act_s0=9.0), dict(activation=1, act_s0=9.0, a_gran=1),
         dict(activation=1, act_s0=9.0, rotation=1), dict(activation=1, act_s0=9.0, rotation=2)]


@pytest.mark.parametrize("kind", range(len(KINDS)))
@pytest.mark.parametrize("width", [64, 128, 256, 512])
def test_small_launches_return_the_observed_kernels_bits(width, kind):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_linear, d_out = (4, 3) if kind % 2 else (8, 2)   # resident and streamed weights at width 256
    dims = (2,) + (width,) * (n_linear - 1) + (d_out,)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 60 + kind)
    grid = to_dev(dhq_inputs.grid_coords(150, 150))
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, **KINDS[kind])
    try:
        dhq.dhq_calibrate(h, grid)
        want = torch.empty((grid.shape[0], d_out), device="cuda")
        dhq.dhq_forward_fused_debug(h, grid, want)
        for n in (1, 31, 64, 65, 129, 1000, sms * 64 - 63, sms * 64, sms * 64 + 1, (sms - 1) * 128 + 1, sms * 128, sms * 128 + 1):
            got = torch.full((n, d_out), float("nan"), device="cuda")
            dhq.dhq_forward(h, grid[:n], got)
            ch, oh = grid[:n].cpu().pin_memory(), torch.zeros((n, d_out)).pin_memory()
            dhq.dhq_forward_host(h, ch, oh)
            torch.cuda.synchronize()
            assert dhq.dhq_last_status(h) == 0
            assert torch.equal(got.view(torch.int32), want[:n].view(torch.int32)), f"n = {n}"
            assert np.array_equal(oh.numpy().view(np.uint32), got.cpu().numpy().view(np.uint32)), f"n = {n}, host buffers"
    finally:
        dhq.dhq_destroy(h)
