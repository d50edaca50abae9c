"""The two-sided transform with a weight scale per output channel, widths 128 and 256: the fixed-point
kernel of dhq_forward at the ends of its tiles and grid, both activation granularities, no and many
tensor-core layers, rows of very different scale (2^-12 to 1 of each other), sine and wavelet.  The
layer-by-layer dumps must satisfy the definition (codes, scales and accumulators exactly, outputs within the
1e-5 of every fused path; measured 7e-7) and dhq_forward must return their bits, since both evaluate
the same exact sums."""
import numpy as np
import pytest
import torch

import dhq_inputs
from tests.gpu_util import check_layers_against_oracle, check_weights, prepare_pair, run_debug, to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")
from oracle import odef  # noqa: E402


@pytest.mark.parametrize("width,n_linear,d_out,a_gran,n,s0", [
    (128, 2, 1, 1, 1, 0.0), (128, 5, 3, 0, 129, 0.0), (128, 4, 2, 1, 148 * 128 + 1, 0.0), (256, 2, 4, 0, 127, 0.0),
    (256, 3, 3, 1, 128, 9.0), (256, 16, 3, 1, 130, 0.0), (256, 4, 3, 0, 148 * 128 + 129, 9.0)])
def test_two_sided_per_channel(width, n_linear, d_out, a_gran, n, s0):
    dims = (2,) + (width,) * (n_linear - 1) + (d_out,)
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 40 + width + n_linear)
    weights[-1] = weights[-1] * np.float32(2.0) ** -np.arange(d_out, dtype=np.float32)[:, None] ** 2
    if n_linear > 2:
        weights[1] = weights[1] * (np.float32(2.0) ** -(np.arange(width) % 13).astype(np.float32))[:, None]
    coords = dhq_inputs.grid_coords(n // 150 + 1, 150)[:n]
    h, net = prepare_pair(dims, weights, biases, 30.0, 8, 8, 1, a_gran, rotate="both", gabor_s0=s0)
    try:
        check_weights(h, net)
        cd = to_dev(coords)
        if a_gran == 0:
            dhq.dhq_calibrate(h, cd)
        dumped, bufs = run_debug(h, net, cd)
        worst = check_layers_against_oracle(h, net, coords, dumped, bufs)
        out = torch.full((n, d_out), float("nan"), device="cuda")
        before = dhq.dhq_launch_count(h)
        dhq.dhq_forward(h, cd, out)
        torch.cuda.synchronize()
        assert dhq.dhq_launch_count(h) - before == 1 and dhq.dhq_last_status(h) == 0
        assert torch.equal(out.view(torch.int32), dumped.view(torch.int32))
        print(f"two-sided per channel, width {width}: outputs within {worst:.2e}")
    finally:
        dhq.dhq_destroy(h)


@pytest.mark.parametrize("width,a_gran,scale", [(128, 1, 1.0), (256, 0, 1.0), (256, 1, 20.0), (128, 0, 300.0)])
def test_phases_are_rounded_once(width, a_gran, scale):
    # The hidden outputs against fp64 on the kernel's own accumulators, phases of 50 to 10,000 rad.  Bound: the hardware
    # sine on [-pi, pi] (2^-21.41 = 3.6e-7) and the phase rounded to fp32 there (half an ulp, 1.2e-7); the entries of a row
    # are multiples of 2^-31 of the largest, so that a sum of them is off by at most that part of the largest phase.
    dims, n = (2, width, width, width, 3), 1500
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 45 + width)
    coords = dhq_inputs.grid_coords(30, 50) * np.float32(scale)
    h, net = prepare_pair(dims, weights, biases, 30.0, 8, 8, 1, a_gran, rotate="both")
    try:
        cd = to_dev(coords)
        dhq.dhq_calibrate(h, cd)
        _, bufs = run_debug(h, net, cd)
        H = odef.hadamard(width)
        worst, excess = [], []
        for l in (1, 2, 3):
            s_w = dhq.dhq_get_layer(h, l)[1].astype(np.float64)
            acc, s_x = bufs["acc"][l - 1].cpu().numpy().astype(np.float64), bufs["s_x"][l - 1].cpu().numpy().astype(np.float64)
            z = (acc * s_w[None, :] * s_x[:, None]) @ H + biases[l - 1].astype(np.float64)[None, :]
            worst.append(np.abs(bufs["Y"][l - 1].cpu().numpy() - np.sin(30.0 * z)).max())
            excess.append(worst[-1] - 2.0 ** -31 * np.abs(30.0 * z).max())
        print(f"two-sided per channel, width {width}, coordinates x {scale}: " + " ".join(f"{x:.2e}" for x in worst))
        assert max(excess) <= 5e-7
    finally:
        dhq.dhq_destroy(h)


@pytest.mark.parametrize("width,a_gran,s0", [(128, 0, 10.0), (256, 1, 10.0), (256, 0, 3.0), (128, 1, 40.0)])
def test_wavelet_envelope_is_rounded_once(width, a_gran, s0):
    # As above for sin(omega0 z) exp(-(s0 z)^2): the sine's bound times the envelope, half an ulp each (6e-8 of the result)
    # for the envelope and the product, and the entries' rounding through both factors (2^-31 of the largest phase).
    dims, n = (2, width, width, width, 3), 1500
    weights, biases = dhq_inputs.siren_init(dims, 30.0, 46 + width)
    coords = dhq_inputs.grid_coords(30, 50)
    h, net = prepare_pair(dims, weights, biases, 30.0, 8, 8, 1, a_gran, rotate="both", gabor_s0=s0)
    try:
        cd = to_dev(coords)
        dhq.dhq_calibrate(h, cd)
        _, bufs = run_debug(h, net, cd)
        H = odef.hadamard(width)
        for l in (1, 2, 3):
            s_w = dhq.dhq_get_layer(h, l)[1].astype(np.float64)
            acc, s_x = bufs["acc"][l - 1].cpu().numpy().astype(np.float64), bufs["s_x"][l - 1].cpu().numpy().astype(np.float64)
            z = (acc * s_w[None, :] * s_x[:, None]) @ H + biases[l - 1].astype(np.float64)[None, :]
            env = np.exp(-(s0 * z) ** 2)
            want = np.sin(30.0 * z) * env
            dz = 2.0 ** -31 * np.abs(z).max()
            bound = 4.8e-7 * env + 1.2e-7 * np.abs(want) + dz * env * (30.0 + 2.0 * s0 * s0 * np.abs(z)) + 1e-37
            err = np.abs(bufs["Y"][l - 1].cpu().numpy() - want)
            print(f"two-sided wavelet, width {width}, s0 {s0}, layer {l}: rms {np.sqrt((err ** 2).mean()):.2e}, of the bound {(err / bound).max():.2f}")
            assert (err <= bound).all()
    finally:
        dhq.dhq_destroy(h)
