"""Floating-point networks whose numbers fixed point would hold with fewer bits than fp32: small activations, weight rows
of wide range, values that are not finite.  They run layer by layer with fp32 multiply-adds; the initialisations the paper's
networks use run in the one-launch kernel.  Bound: the rms error of a layer's outputs relative to theirs that
fp32 sums of K products show, 0.6 sqrt(K) 2^-24 for phases of order 1, and 1.5e-7 for the hardware sine (fixed point: 3e-6
with activations of 0.03, 1.5e-4 with a dominant weight on an input that is zero)."""
import numpy as np
import pytest
import torch

import dhq_inputs
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

dhq = pytest.importorskip("paper_2508_13478_b200")
from oracle import odef  # noqa: E402


def _network(kind, width, n_hidden=3):
    dims = (2,) + (width,) * n_hidden + (3,)
    W, B = dhq_inputs.siren_init(dims, 30.0, 11)
    if kind == "trained":
        W, B = dhq_inputs.trained_like_init(dims, 30.0, 11)
    elif kind.startswith("small"):                  # the second layer's phases stay of order 1
        r = np.float32(float(kind[5:]))
        W[0], B[0], W[1] = W[0] * (r / 15), B[0] * (r / 15), W[1] / r
    elif kind == "no bias":
        B = [np.zeros_like(b) for b in B]
    elif kind == "wide rows":                       # one weight 12 times the others' rms
        s = np.float32(np.sqrt(2.0 / width) / 30.0)
        W[1] = W[1] / s
        W[1][np.arange(width), (7 * np.arange(width)) % width] = 12.0
        W[1] = (W[1] / np.sqrt((W[1] ** 2).mean(1, keepdims=True)) * s).astype(np.float32)
    elif kind == "one wide row":
        W[1][5, 9] = 3.0
    elif kind == "dominant":                        # on an input that is zero throughout
        W[0][7], B[0][7], W[1][:, 7] = 0.0, 0.0, 10.0
    return dims, W, B


def _prepare(dims, W, B, w_bits):
    return dhq.dhq_prepare(dims, [to_dev(x) for x in W], [to_dev(x) for x in B], 30.0, w_bits, dhq.DHQ_BITS_FLOAT)


@pytest.mark.parametrize("kind,width,w_bits,one_launch", [
    ("default", 64, 32, True), ("default", 64, 8, True), ("default", 512, 8, True), ("trained", 128, 32, True), ("trained", 256, 32, True),
    ("trained", 512, 8, True), ("small0.03", 64, 32, False), ("small0.03", 256, 32, False), ("small0.03", 256, 8, False),
    ("small0.1", 512, 8, False), ("small0.001", 128, 32, False), ("no bias", 256, 32, False), ("wide rows", 64, 32, False),
    ("wide rows", 256, 32, False), ("one wide row", 256, 32, False), ("dominant", 128, 32, False), ("dominant", 512, 32, False)])
def test_error_and_route(kind, width, w_bits, one_launch):
    dims, W, B = _network(kind, width)
    n = 1000 + 37
    coords = (np.random.default_rng(5).random((n, 2)) * 2 - 1).astype(np.float32)
    h = _prepare(dims, W, B, w_bits)
    try:
        cd = to_dev(coords)
        X = [torch.empty((n, dhq.dhq_layer_dims(h, l)[0]), device="cuda") for l in range(1, 5)]
        Y = [torch.empty((n, dhq.dhq_layer_dims(h, l)[1]), device="cuda") for l in range(1, 5)]
        dumped, out = torch.empty((n, 3), device="cuda"), torch.full((n, 3), float("nan"), device="cuda")
        dhq.dhq_forward_debug(h, cd, dumped, {"X": X, "Y": Y})
        before = dhq.dhq_launch_count(h)
        dhq.dhq_forward(h, cd, out)
        assert dhq.dhq_launch_count(h) - before == (1 if one_launch else 4)
        oh = torch.zeros((n, 3)).pin_memory()
        dhq.dhq_forward_host(h, torch.from_numpy(coords).pin_memory(), oh)
        blob = dhq.dhq_export(h)
        h2 = dhq.dhq_import(blob)
        try:
            assert dhq.dhq_export(h2) == blob
            out2 = torch.full_like(out, float("nan"))
            dhq.dhq_forward(h2, cd, out2)
            torch.cuda.synchronize()
        finally:
            dhq.dhq_destroy(h2)
        assert dhq.dhq_last_status(h) == 0
        for other in (dumped, out2, oh.cuda()):
            assert torch.equal(out.view(torch.int32), other.view(torch.int32))
        layers = [dhq.dhq_get_layer(h, l) for l in (1, 2, 3)]
    finally:
        dhq.dhq_destroy(h)
    for l in (2, 3):
        x = X[l - 1].cpu().numpy()
        if w_bits < 32:
            want = odef.w8a32_layer(layers[l - 1][0], layers[l - 1][1], B[l - 1], x, True, 30.0, True)
        else:
            want = np.sin(30.0 * (x.astype(np.float64) @ W[l - 1].astype(np.float64).T + B[l - 1].astype(np.float64)))
        rel = np.linalg.norm(Y[l - 1].cpu().numpy() - want) / np.linalg.norm(want)
        phase = 30.0 * np.sqrt((W[l - 1].astype(np.float64) ** 2).sum(1).mean() * (x.astype(np.float64) ** 2).mean())
        print(f"W{w_bits}A32 {kind} width {width} layer {l}: {rel:.2e}, phases {phase:.1f}")
        if kind != "dominant":
            assert rel <= max(1.0, phase) * 0.6 * np.sqrt(width) * 2.0 ** -24 + 1.5e-7
        else:                                       # (the rms of the weights says nothing here)
            assert rel <= 0.6 * np.sqrt(width) * 2.0 ** -24 + 1.5e-7


@pytest.mark.parametrize("w_bits", [32, 8])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_weights_that_are_not_finite_reach_the_result(w_bits, value):
    dims, W, B = _network("default", 128)
    for where in ("weight", "bias", "last"):
        w, b = [x.copy() for x in W], [x.copy() for x in B]
        if where == "weight":
            w[1][3, 4] = value
        elif where == "bias":
            b[2][0] = value
        else:
            w[3][0, 0] = value
        if w_bits == 8 and where != "bias":
            continue                                # the weight quantizer makes what it makes of them
        h = _prepare(dims, w, b, w_bits)
        try:
            out = torch.zeros((300, 3), device="cuda")
            dhq.dhq_forward(h, to_dev(dhq_inputs.grid_coords(3, 100)), out)
            torch.cuda.synchronize()
            assert dhq.dhq_last_status(h) == 0
            assert not torch.isfinite(out[:, 0]).any()
        finally:
            dhq.dhq_destroy(h)


@pytest.mark.parametrize("width,w_bits,n_hidden", [(64, 32, 3), (128, 8, 2), (256, 32, 1), (512, 8, 3)])
def test_coordinates_that_are_not_finite_reach_the_result(width, w_bits, n_hidden):
    dims, W, B = _network("default", width, n_hidden)
    coords = dhq_inputs.grid_coords(200, 150)
    bad = coords.copy()
    rows = np.arange(5, len(bad), 997)
    bad[rows, rows % 2] = np.where(rows % 3 == 0, np.nan, np.where(rows % 3 == 1, np.inf, -np.inf)).astype(np.float32)
    h = _prepare(dims, W, B, w_bits)
    try:
        out, want = torch.zeros((len(bad), 3), device="cuda"), torch.zeros((len(bad), 3), device="cuda")
        dhq.dhq_forward(h, to_dev(coords), want)
        dhq.dhq_forward(h, to_dev(bad), out)
        torch.cuda.synchronize()
        assert dhq.dhq_last_status(h) == 0
    finally:
        dhq.dhq_destroy(h)
    got, want = out.cpu().numpy(), want.cpu().numpy()
    assert np.isnan(got[rows]).all()
    rest = np.setdiff1d(np.arange(len(bad)), rows)
    assert np.array_equal(got[rest].view(np.uint32), want[rest].view(np.uint32))
