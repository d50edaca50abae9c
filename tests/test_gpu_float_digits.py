"""The floating-point datapaths where their fixed-point kernel can go wrong: every width, one and
several tiles with ragged ends, more tiles than the grid has blocks, no tensor-core layer (L = 2),
many layers, and integer rows that need a third digit (a weight row with one dominant input: its
rotated codes are +-127 throughout, so q H has an entry of 127 K).

The reference is the fp64 definition of each layer on the library's own input of that layer, at the
gate of the other float tests: fp32 phase of the first layer (50 rad, half an ulp 1.9e-6, and the
rounding of its constants, 3e-6), 24-bit activations and weights of the others (below 2e-6)."""
import numpy as np
import pytest
import torch

import dhq_inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")
from oracle import dhq_oracle as orc  # noqa: E402
from oracle import odef  # noqa: E402

TOL_FLOAT = 2e-5


@pytest.mark.parametrize("width,n_linear,d_out,n,w_bits,sparse", [
    (64, 2, 1, 1, 32, False), (64, 5, 4, 127, 8, False), (128, 3, 2, 129, 32, False), (128, 4, 3, 300, 8, True),
    (256, 16, 3, 128, 32, False), (256, 3, 1, 128 * 149 + 5, 8, False), (256, 4, 4, 257, 8, True), (512, 2, 3, 200, 8, False),
    (512, 3, 3, 128 * 148 + 1, 32, False), (512, 4, 2, 385, 8, True), (512, 5, 3, 1, 4, False)])
def test_fixed_point_layers(width, n_linear, d_out, n, w_bits, sparse):
    dims = (2,) + (width,) * (n_linear - 1) + (d_out,)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 700 + width + n_linear)
    if sparse:
        weights[1][::3] = 0.0
        weights[1][np.arange(0, width, 3), (7 * np.arange(0, width, 3)) % width] = 0.02
    coords = dhq_inputs.grid_coords(n // 100 + 1, 100)[:n]
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, w_bits, dhq.DHQ_BITS_FLOAT)
    try:
        cd = to_dev(coords)
        X = [torch.empty((n, dhq.dhq_layer_dims(h, l)[0]), device="cuda") for l in range(1, n_linear + 1)]
        Y = [torch.empty((n, dhq.dhq_layer_dims(h, l)[1]), device="cuda") for l in range(1, n_linear + 1)]
        dumped = torch.empty((n, d_out), device="cuda")
        dhq.dhq_forward_debug(h, cd, dumped, {"X": X, "Y": Y})
        out = torch.full((n, d_out), float("nan"), device="cuda")
        dhq.dhq_forward(h, cd, out)
        torch.cuda.synchronize()
        assert dhq.dhq_last_status(h) == 0
        assert torch.equal(out.view(torch.int32), dumped.view(torch.int32))
    finally:
        dhq.dhq_destroy(h)
    net = orc.prepare(weights, biases, dims, 30.0, w_bits if w_bits < 32 else 8, 8, 0, 1, rotate=True)
    for l in range(1, n_linear + 1):
        x = X[l - 1].cpu().numpy()
        if w_bits < 32:
            lay = net.layers[l - 1]
            want = odef.w8a32_layer(lay.qw, lay.s_w, lay.b_pad, x, True, 30.0, lay.sine)
        else:
            z = x.astype(np.float64)[:, : dims[l - 1]] @ weights[l - 1].astype(np.float64).T + biases[l - 1].astype(np.float64)
            want = np.sin(30.0 * z) if l < n_linear else z
        got = Y[l - 1].cpu().numpy()[:, : want.shape[1]]
        assert np.abs(got - want).max() <= TOL_FLOAT, f"layer {l}"


@pytest.mark.parametrize("width,n_linear", [(64, 3), (128, 3), (64, 2), (128, 4), (256, 3)])
def test_tiles_of_one_block_do_not_disturb_each_other(width, n_linear):
    # several tiles per block of the grid: the next tile's last-layer sums must not reach the columns of this tile's
    # (the ordering differs with the number of layers and of output blocks); every tile alone gives the bits to expect
    dims = (2,) + (width,) * (n_linear - 1) + (3,)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 900 + width + n_linear)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 128 * (3 * sms + 1) + 77
    cd = to_dev(dhq_inputs.grid_coords(n // 240 + 1, 240)[:n])
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, 32, dhq.DHQ_BITS_FLOAT)
    try:
        want = torch.empty((n, 3), device="cuda")
        for t in range(0, n, 128 * sms):   # one tile per block
            dhq.dhq_forward(h, cd[t:t + 128 * sms], want[t:t + 128 * sms])
        for _ in range(20):
            got = torch.full((n, 3), float("nan"), device="cuda")
            dhq.dhq_forward(h, cd, got)
            assert torch.equal(got.view(torch.int32), want.view(torch.int32))
        assert dhq.dhq_last_status(h) == 0
    finally:
        dhq.dhq_destroy(h)


@pytest.mark.parametrize("n_linear,w_bits", [(3, 32), (3, 8), (4, 8), (6, 32)])
def test_tiles_of_one_block_at_width_512(n_linear, w_bits):
    # the same for the width whose third digit, constants and last-layer sums pass from tile to tile through tensor and
    # shared memory: one and several tensor-core layers, two and three weight digits
    dims = (2,) + (512,) * (n_linear - 1) + (3,)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 950 + n_linear)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 128 * (2 * sms + 1) + 77
    cd = to_dev(dhq_inputs.grid_coords(n // 240 + 1, 240)[:n])
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, w_bits, dhq.DHQ_BITS_FLOAT)
    try:
        want = torch.empty((n, 3), device="cuda")
        for t in range(0, n, 128 * sms):   # one tile per block
            dhq.dhq_forward(h, cd[t:t + 128 * sms], want[t:t + 128 * sms])
        for _ in range(5):
            got = torch.full((n, 3), float("nan"), device="cuda")
            dhq.dhq_forward(h, cd, got)
            assert torch.equal(got.view(torch.int32), want.view(torch.int32))
        assert dhq.dhq_last_status(h) == 0
    finally:
        dhq.dhq_destroy(h)


@pytest.mark.parametrize("width", [64, 256, 512])
def test_dump_buffers_and_coordinates_need_no_more_than_float_alignment(width):
    dims, n = (2, width, width, width, 3), 300
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 950 + width)
    coords = to_dev(dhq_inputs.grid_coords(3, 100))
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, 32, dhq.DHQ_BITS_FLOAT)
    try:
        def run(shift):  # every buffer `shift` floats past a 256-byte boundary
            def buf(cols):
                return torch.full((n * cols + 4,), float("nan"), device="cuda")[shift:shift + n * cols].view(n, cols)
            X = [buf(dhq.dhq_layer_dims(h, l)[0]) for l in range(1, 5)]
            Y = [buf(dhq.dhq_layer_dims(h, l)[1]) for l in range(1, 5)]
            c, out = buf(2), buf(3)
            c.copy_(coords)
            dhq.dhq_forward_debug(h, c, out, {"X": X, "Y": Y})
            torch.cuda.synchronize()
            assert dhq.dhq_last_status(h) == 0
            return X + Y + [out]
        for got, want in zip(run(1), run(0)):
            assert torch.equal(got.view(torch.int32), want.view(torch.int32))
    finally:
        dhq.dhq_destroy(h)


@pytest.mark.parametrize("width,w_bits,hidden", [(64, 32, 2.1e-7), (64, 8, 2.2e-7), (128, 32, 2.5e-7), (128, 8, 2.6e-7), (256, 32, 3.2e-7),
                                                 (256, 8, 3.2e-7), (512, 32, 4.2e-7), (512, 8, 4.3e-7)])
def test_no_less_exact_than_fp32_multiply_adds(width, w_bits, hidden):
    # rms error of a layer's outputs relative to their rms, against fp64 on the kernel's own inputs of the layer.  Bounds: what
    # fp32 multiply-adds with an fp32 phase give for these networks (5.6e-7 for the first layer).
    dims, n = (2, width, width, width, 3), 2048
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 11)
    coords = np.ascontiguousarray(np.random.default_rng(5).random((n, 2)) * 2 - 1).astype(np.float32)
    h = dhq.dhq_prepare(dims, [to_dev(x) for x in weights], [to_dev(x) for x in biases], 30.0, w_bits, dhq.DHQ_BITS_FLOAT)
    try:
        X = [torch.empty((n, dhq.dhq_layer_dims(h, l)[0]), device="cuda") for l in range(1, 5)]
        Y = [torch.empty((n, dhq.dhq_layer_dims(h, l)[1]), device="cuda") for l in range(1, 5)]
        dhq.dhq_forward_debug(h, to_dev(coords), None, {"X": X, "Y": Y})
        torch.cuda.synchronize()
        layers = [dhq.dhq_get_layer(h, l) for l in (1, 2, 3)]
    finally:
        dhq.dhq_destroy(h)
    for l, (codes, scales, _) in enumerate(layers, start=1):
        x = X[l - 1].cpu().numpy()
        if w_bits < 32:
            want = odef.w8a32_layer(codes, scales, biases[l - 1], x, True, 30.0, True)
        else:
            want = np.sin(30.0 * (x.astype(np.float64)[:, : dims[l - 1]] @ weights[l - 1].astype(np.float64).T + biases[l - 1].astype(np.float64)))
        rel = np.linalg.norm(Y[l - 1].cpu().numpy() - want) / np.linalg.norm(want)
        print(f"W{w_bits}A32 width {width} layer {l}: {rel:.2e}")
        assert rel <= (5.6e-7 if l == 1 else hidden)
