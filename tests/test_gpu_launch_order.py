"""Order of launches: forwards set themselves up beside the launch before them, and the calibration passes do the
same.  Whatever precedes a forward in its stream - calibration, a forward in another stream, a captured one, the forward
that writes its coordinates - it must give the bits of a call made on an idle device."""
import pytest
import torch

import dhq_inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")


def _network(width, d_out, seed, **kw):
    dims = (2, width, width, width, width, d_out)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, seed)
    return dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, **kw)


def _alone(h, coords, d_out):
    out = torch.empty((coords.shape[0], d_out), device="cuda")
    torch.cuda.synchronize()
    dhq.dhq_forward(h, coords, out)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("width", [64, 128, 256, 512])
@pytest.mark.parametrize("between", ["nothing", "other_stream", "capture"])
def test_forward_directly_behind_a_calibration(width, between):
    h = _network(width, 3, 300 + width)
    try:
        # a few tiles only: blocks of the forward find SMs beside the calibration passes
        small, other = to_dev(dhq_inputs.grid_coords(40, 50)), to_dev(dhq_inputs.grid_coords(30, 61)) * 0.25
        side = torch.cuda.Stream()
        want = {}
        for name, c in (("small", small), ("other", other)):
            dhq.dhq_calibrate(h, c)
            want[name] = _alone(h, c, 3)
        assert not torch.equal(want["small"][:100], want["other"][:100])
        for i in range(30):
            name, c = (("small", small), ("other", other))[i & 1]
            first, got = torch.empty_like(want[name]), torch.full_like(want[name], float("nan"))
            torch.cuda.synchronize()
            dhq.dhq_calibrate(h, c)
            if between == "other_stream":
                side.wait_stream(torch.cuda.current_stream())
                dhq.dhq_forward(h, c, first, stream=side)
            elif between == "capture":
                side.wait_stream(torch.cuda.current_stream())
                graph = torch.cuda.CUDAGraph()
                # (relaxed: allocations and destructions of other objects stay allowed meanwhile)
                with torch.cuda.graph(graph, stream=side, capture_error_mode="relaxed"):
                    dhq.dhq_forward(h, c, first)
            dhq.dhq_forward(h, c, got)
            torch.cuda.synchronize()
            assert torch.equal(got.view(torch.int32), want[name].view(torch.int32)), f"pass {i}"
            if between == "other_stream":
                assert torch.equal(first.view(torch.int32), want[name].view(torch.int32)), f"pass {i}, other stream"
            elif between == "capture":
                graph.replay()
                torch.cuda.synchronize()
                assert torch.equal(first.view(torch.int32), want[name].view(torch.int32)), f"pass {i}, replay"
        assert dhq.dhq_last_status(h) == 0
    finally:
        dhq.dhq_destroy(h)


@pytest.mark.parametrize("width,kw", [(64, dict()), (256, dict()), (512, dict()), (256, dict(w_gran=1, a_gran=1, rotation=1)),
                                      (128, dict(w_bits=32, a_bits=32)), (512, dict(w_bits=32, a_bits=32))])
@pytest.mark.parametrize("n", [100, 5000, 40000])
def test_a_forward_reads_what_the_one_before_it_wrote(width, kw, n):
    # two outputs used as the next call's coordinates, back to back
    h = _network(width, 2, 400 + width, **kw)
    try:
        c = to_dev(dhq_inputs.grid_coords(n // 100, 100))
        dhq.dhq_calibrate(h, c)
        want, x = [], c
        for _ in range(6):
            x = _alone(h, x, 2)
            want.append(x)
        bufs = [torch.full_like(c, float("nan")) for _ in range(6)]
        torch.cuda.synchronize()
        x = c
        for b in bufs:
            dhq.dhq_forward(h, x, b)
            x = b
        a, b = c.clone(), torch.empty_like(c)      # and in two buffers, each overwritten while the launch behind is set up
        for _ in range(3):
            dhq.dhq_forward(h, a, b)
            dhq.dhq_forward(h, b, a)
        torch.cuda.synchronize()
        for i in range(6):
            assert torch.equal(bufs[i].view(torch.int32), want[i].view(torch.int32)), f"step {i}"
        assert torch.equal(a.view(torch.int32), want[5].view(torch.int32))
        assert dhq.dhq_last_status(h) == 0
    finally:
        dhq.dhq_destroy(h)
