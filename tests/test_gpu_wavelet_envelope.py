"""The wavelet exp(-(s0 z)^2) sin(omega0 z) where its envelope is below 2^-126: results there keep the bits that fp32 has
for them, on the layer-by-layer route and inside the fused kernel."""
import numpy as np
import pytest
import torch

import dhq_inputs
from tests.gpu_util import prepare_pair, run_debug, to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("width,a_gran,rotate", [(64, 0, True), (64, 1, True), (128, 0, False), (256, 1, False), (256, 0, True), (512, 1, True)])
def test_subnormal_envelopes_are_not_zero(width, a_gran, rotate, fused):
    s0, omega0, dims = 2.0, 30.0, (2, width, width, 3)
    rng = np.random.default_rng(81)
    weights = [rng.uniform(-3.0, 3.0, (width, 2)), rng.normal(0.0, 8.0 / width ** 0.5, (width, width)), rng.uniform(-0.1, 0.1, (3, width))]
    biases = [rng.uniform(-1.0, 1.0, w.shape[0]) for w in weights]
    weights, biases = [w.astype(np.float32) for w in weights], [b.astype(np.float32) for b in biases]
    h, net = prepare_pair(dims, weights, biases, omega0, 8, 8, a_gran, a_gran, rotate=rotate, gabor_s0=s0)
    try:
        cd = to_dev(dhq_inputs.grid_coords(50, 61))
        dhq.dhq_calibrate(h, cd)
        _, bufs = run_debug(h, net, cd, fused=fused)
        for l in (1, 2):
            s_x = bufs["s_x"][l - 1].cpu().numpy().astype(np.float64)[:, None]
            z = net.layers[l - 1].s_w.astype(np.float64)[None, :] * s_x * bufs["acc"][l - 1].cpu().numpy() + biases[l - 1].astype(np.float64)[None, :]
            envelope = np.exp(-(s0 * z) ** 2)
            want = np.sin(omega0 * z) * envelope
            got = bufs["Y"][l - 1].cpu().numpy().astype(np.float64)
            few = (envelope < 2.0 ** -126) & (envelope >= 2.0 ** -149)
            assert few.sum() > 200, "the network does not meet the range"
            # The exponent, at most 149 ln 2 = 103.3, is a square with the phase's relative error (at most 3 * 2^-24) twice, and
            # two products and a constant rounded to fp32: 103.3 * 9 * 2^-24 = 5.6e-5, ex2.approx's 2^-22 and the sine's 1e-5 beside
            # it; the envelope and the product are each rounded to a multiple of 2^-149.
            bound = 6.7e-5 * envelope + 2.0 ** -148
            err = np.abs(got - want)[few]
            print(f"width {width}, layer {l}: {few.sum()} results, largest error {(err / bound[few]).max():.2f} of the bound")
            assert (err <= bound[few]).all()
            assert (got[few] != 0.0).sum() > 100
    finally:
        dhq.dhq_destroy(h)
