"""The bounded waits of the floating-point kernel and of the two-sided per-channel kernel: with one copy of weights left out
(nothing is in flight for it) every role gives up after the handle's wait limit, the kernel frees its tensor memory and
returns, the status word says TIMEOUT, and the next launch gives the bits of the one before."""
import pytest
import torch

import dhq_inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")

DIGITS = dict(w_gran=1, rotation=1)


@pytest.mark.parametrize("width,kw,n", [(64, dict(w_bits=32, a_bits=32), 100), (256, dict(w_bits=8, a_bits=32), 100), (512, dict(w_bits=32, a_bits=32), 100),
                                        (512, dict(w_bits=8, a_bits=32), 40000), (128, DIGITS, 100), (256, dict(a_gran=1, **DIGITS), 40000)])
def test_a_wait_that_runs_out_is_reported_and_the_handle_stays_usable(width, kw, n):
    dims = (2, width, width, width, 3)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 17)
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, **kw)
    try:
        cd = to_dev(dhq_inputs.grid_coords(n // 100, 100))
        dhq.dhq_calibrate(h, cd)
        ref = torch.empty((n, 3), device="cuda")
        dhq.dhq_forward(h, cd, ref)
        torch.cuda.synchronize()
        assert dhq.dhq_last_status(h) == 0
        dhq.dhq_set_wait_limit(h, 5_000_000)                       # 5 ms
        dhq.dhq_debug_stall_next_forward(h)
        junk = torch.zeros_like(ref)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        dhq.dhq_forward(h, cd, junk)
        t1.record()
        torch.cuda.synchronize()
        assert t0.elapsed_time(t1) < 500.0                         # milliseconds
        assert dhq.dhq_last_status(h) == 6                         # DHQ_ERR_TIMEOUT
        assert dhq.dhq_last_status(h) == 0
        out = torch.zeros_like(ref)
        dhq.dhq_forward(h, cd, out)
        torch.cuda.synchronize()
        assert dhq.dhq_last_status(h) == 0
        assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    finally:
        dhq.dhq_destroy(h)


def test_the_hook_is_refused_where_no_weights_are_copied():
    dims = (2, 64, 3)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 17)
    for options in (dict(w_bits=32, a_bits=32), dict(w_gran=1, rotation=1)):
        h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, **options)
        try:
            with pytest.raises(dhq.DhqError) as e:
                dhq.dhq_debug_stall_next_forward(h)
            assert e.value.code == 2
        finally:
            dhq.dhq_destroy(h)
