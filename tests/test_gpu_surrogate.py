"""GPU parity of the learned surrogate's BF16 tensor-core kernels against the FP64 MLP
oracle (forward, gradients, Adam), its inputs against the dynamics oracle, and the
surrogate control step: its one-step error against the plain integrator, what the network
gains over predicting no change, and the out-of-distribution fallback."""
import hashlib
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import paper_2606_08039_gb300 as mdg
from oracle import mlp as omlp
from paper_2606_08039_gb300 import surrogate as sg
from paper_2606_08039_gb300 import workloads as wl
from helpers import assert_horizon_close, assert_knn_valid, check_obs_against_own_state, excess, oracle_arrays, oracle_step, \
    spread_heights, tolerance_response

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
P = oracle.cf2x()
HOVER = oracle.hover_rpm(P)


def _layers(seed, bias_scale=0.1):
    layers = wl.mlp_init(seed)
    out = []
    for l, (W, b) in enumerate(layers):
        bb = wl.uniform_range(-bias_scale, bias_scale, seed, wl.S_MLP, 100 + l, np.arange(b.size, dtype=np.uint64), 0)
        out.append((W, bb))
    return out


def _inputs(seed, B):
    x = np.zeros((B, mdg.MLP_IN_PAD), np.float32)
    x[:, :mdg.MLP_IN] = wl.uniform_range(-2, 2, seed, 11, 0, np.arange(B, dtype=np.uint64)[:, None],
                                         np.arange(mdg.MLP_IN, dtype=np.uint64)[None, :])
    return x


def _tanh_error_response(params, x, y_ref, rel=2.0 ** -11):
    """|change of the oracle's output| when every tanh inside SiLU = z/2 (1 + tanh(z/2))
    carries a relative error of `rel` (random signs)."""
    rng = np.random.default_rng(0)
    exact = omlp.silu

    def perturbed(z):
        return 0.5 * z * (1.0 + np.tanh(z / 2) * (1.0 + rel * rng.choice([-1.0, 1.0], size=np.shape(z))))
    omlp.silu = perturbed
    try:
        yp, _ = omlp.forward(params, x, bf16_storage=True)
    finally:
        omlp.silu = exact
    return np.abs(yp - y_ref)


def _f64(layers):
    return [(np.asarray(W, np.float64), np.asarray(b, np.float64)) for W, b in layers]


@pytest.mark.parametrize("path,B", [(mdg.MLP_PATH_TCGEN05, 128), (mdg.MLP_PATH_TCGEN05, 384 * 8),
                                    (mdg.MLP_PATH_MMA_SYNC, 384), (mdg.MLP_PATH_TCGEN05_PAIRS, 128),
                                    (mdg.MLP_PATH_TCGEN05_PAIRS, 384 * 8)])
def test_forward_matches_oracle(cuda, path, B):
    """The inference paths (fused tcgen05 kernel, its two-tiles-in-flight form, per-layer
    mma.sync GEMMs) against the oracle on identical bf16 inputs and weights; several tiles per
    block for the persistent tcgen05 kernels, and for the paired one a lone tile."""
    layers = _layers(1)
    m = mdg.MLP(B, layers)
    m.set_path(path)
    x = torch.as_tensor(_inputs(2, B), device=cuda).to(torch.bfloat16)
    y = torch.full((B, mdg.MLP_OUT_PAD), float("nan"), device=cuda)
    m.forward(x, y)
    torch.cuda.synchronize()
    assert m.status() == 0
    xo = x.float().cpu().numpy().astype(np.float64)
    yo, _ = omlp.forward(_f64(layers), xo, bf16_storage=True)
    # identical bf16 inputs and weights; FP32 vs FP64 accumulation can flip the bf16 rounding
    # of a hidden activation by one bf16 unit (2^-8 relative), hence 1e-2 max(|y|, 1). The
    # tcgen05 path evaluates SiLU as z/2 (1 + tanh(z/2)) with tanh.approx.f32 (relative error
    # 2^-11): its bound adds the oracle's own response to that error.
    bound = 1e-2 * np.maximum(np.abs(yo), 1.0)
    if path != mdg.MLP_PATH_MMA_SYNC:
        bound = bound + _tanh_error_response(_f64(layers), xo, yo)
    assert np.all(np.abs(y.cpu().numpy() - yo) <= bound)


def test_training_paths_agree_over_steps(cuda):
    """Eight Adam steps on the tcgen05 path and on the mma.sync path from the same weights and
    batches: losses within 1% and the weights within 10% of their change (accumulation order
    and bf16 rounding of the stored activations differ, and Adam's first steps move a weight
    by about lr whatever the size of its gradient, so the sign of a near-zero gradient
    matters)."""
    B = 512
    layers = _layers(7)
    x = torch.as_tensor(_inputs(8, B), device=cuda).to(torch.bfloat16)
    t = torch.zeros((B, mdg.MLP_OUT_PAD), device=cuda)
    t[:, :mdg.MLP_OUT] = torch.as_tensor(
        wl.uniform_range(-1, 1, 9, 12, 0, np.arange(B, dtype=np.uint64)[:, None],
                         np.arange(mdg.MLP_OUT, dtype=np.uint64)[None, :]), device=cuda)
    w0 = mdg.mlp_flatten(layers).astype(np.float64)
    out = []
    for path in (mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_MMA_SYNC):
        m = mdg.MLP(B, layers)
        m.set_train_path(path)
        loss = torch.zeros(1, device=cuda)
        losses = []
        for _ in range(8):
            m.grad(x, t, loss)
            losses.append(float(loss))
            m.adam(1e-3)
        torch.cuda.synchronize()
        assert m.status() == 0
        out.append((np.array(losses), m.params().astype(np.float64)))
    (la, wa), (lb, wb) = out
    np.testing.assert_allclose(la, lb, rtol=1e-2)
    assert la[-1] < la[0]
    dw = np.abs(wb - w0)
    assert np.linalg.norm(wa - wb) <= 0.1 * np.linalg.norm(dw)


@pytest.mark.parametrize("path", [mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_TCGEN05_PAIRS])
def test_tcgen05_bounded_wait_exit(cuda, path):
    """The tcgen05 kernel's exit on an expired wait, without a stuck device: with wait bounds
    of zero the first wait that is not already complete (at the latest the epilogue's wait
    for its first accumulator) gives up on a normal 256-row launch, in both tcgen05 kernels. The launch returns with
    MDG_STATUS_TIMEOUT set; a launch with the default bounds then matches the oracle, so the
    abandoned launch drained its copies and MMAs and freed its tensor memory."""
    layers = _layers(1)
    B = 256  # one pair of tiles for the paired kernel
    m = mdg.MLP(B, layers)
    m.set_path(path)
    x = torch.as_tensor(_inputs(2, B), device=cuda).to(torch.bfloat16)
    y = torch.full((B, mdg.MLP_OUT_PAD), float("nan"), device=cuda)
    m.set_wait_limits(0, 0)
    m.forward(x, y)
    assert mdg.lib().mdg_sync(mdg._stream(None), 5000) == mdg.OK  # the launch returned
    assert m.status() & mdg.STATUS_TIMEOUT
    for _ in range(2):  # again, and on the blocks' second use of the SMs' tensor memory
        m.forward(x, y)
        torch.cuda.synchronize()
        assert m.status() & mdg.STATUS_TIMEOUT
    m.set_wait_limits()
    y.fill_(float("nan"))
    m.forward(x, y)
    torch.cuda.synchronize()
    assert m.status() == 0
    xo = x.float().cpu().numpy().astype(np.float64)
    yo, _ = omlp.forward(_f64(layers), xo, bf16_storage=True)
    bound = 1e-2 * np.maximum(np.abs(yo), 1.0) + _tanh_error_response(_f64(layers), xo, yo)
    assert np.all(np.abs(y.cpu().numpy() - yo) <= bound)


@pytest.mark.parametrize("n_tiles", [305, 611])
def test_paired_kernel_equals_single_tile_kernel(cuda, n_tiles):
    """The two-tiles-in-flight kernel does the first tile of each pair (A, even tiles) exactly
    as the single-tile kernel (the same MMAs in the same order, the same epilogue per element),
    so those outputs are bit-identical; the second tile (B) sums the K chunks of its hidden
    layers in the order 3, 2, 1, 0, so it agrees to FP32 summation order (and the bf16
    rounding that follows). Here with two to three pairs per block and a lone last tile (305
    tiles: 153 pairs on 152 SMs; 611 tiles); and sampled tiles of it against the oracle."""
    B = 128 * n_tiles
    layers = _layers(4)
    m = mdg.MLP(B, layers)
    x = torch.as_tensor(_inputs(6, B), device=cuda).to(torch.bfloat16)
    ys = []
    for path in (mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_TCGEN05_PAIRS):
        m.set_path(path)
        y = torch.full((B, mdg.MLP_OUT_PAD), float("nan"), device=cuda)
        m.forward(x, y)
        torch.cuda.synchronize()
        assert m.status() == 0
        ys.append(y)
    single, paired = (y.view(n_tiles, 128, mdg.MLP_OUT_PAD) for y in ys)
    assert torch.equal(single[0::2], paired[0::2])
    assert torch.all((single[1::2] - paired[1::2]).abs() <= 1e-2 * torch.clamp(single[1::2].abs(), min=1.0))
    tiles = [0, 1, 151, 152, 153, 303, 304, n_tiles - 2, n_tiles - 1]
    rows = np.concatenate([np.arange(128 * t, 128 * t + 128) for t in sorted(set(tiles))])
    xo = x[torch.as_tensor(rows, device=cuda)].float().cpu().numpy().astype(np.float64)
    yo, _ = omlp.forward(_f64(layers), xo, bf16_storage=True)
    bound = 1e-2 * np.maximum(np.abs(yo), 1.0) + _tanh_error_response(_f64(layers), xo, yo)
    assert np.all(np.abs(ys[1].cpu().numpy()[rows] - yo) <= bound)


@pytest.mark.parametrize("n_tiles", [1, 2, 152, 153, 303, 304, 305, 340, 456, 457])
def test_lone_last_tiles(cuda, n_tiles):
    """The tiles left after the whole rounds of pairs, alone on a block each or in one more round of
    pairs (152 SMs: the rule changes at 152 tiles left): a lone tile runs as the first of a pair, so
    it equals the single-tile kernel's, as every even tile does; the others to the summation order's
    bound of the test above."""
    B, sms = 128 * n_tiles, torch.cuda.get_device_properties(0).multi_processor_count
    m = mdg.MLP(B, _layers(4))
    x = torch.as_tensor(_inputs(7, B), device=cuda).to(torch.bfloat16)
    ys = []
    for path in (mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_TCGEN05_PAIRS):
        m.set_path(path)
        y = torch.full((B, mdg.MLP_OUT_PAD), float("nan"), device=cuda)
        m.forward(x, y)
        assert m.status() == 0
        ys.append(y.view(n_tiles, 128, mdg.MLP_OUT_PAD))
    first = np.arange(n_tiles) % 2 == 0
    whole = n_tiles // (2 * sms) * 2 * sms
    if n_tiles - whole <= sms:
        first[whole:] = True
    first = torch.as_tensor(first, device=cuda)
    assert torch.equal(ys[0][first], ys[1][first])
    assert torch.all((ys[0] - ys[1]).abs() <= 1e-2 * torch.clamp(ys[0].abs(), min=1.0))


@pytest.mark.parametrize("path,B", [(mdg.MLP_PATH_TCGEN05, 256), (mdg.MLP_PATH_TCGEN05, 1024),
                                    (mdg.MLP_PATH_MMA_SYNC, 256)])
def test_gradients_and_loss_match_oracle(cuda, path, B):
    """Loss and every gradient of both training paths (tcgen05 with TMEM accumulators, the
    default; mma.sync) against the FP64 oracle's backward on the same bf16 tensors; B = 1024
    splits the weight gradients over the batch (two slices added with atomics)."""
    layers = _layers(3)
    m = mdg.MLP(B, layers)
    m.set_train_path(path)
    x = torch.as_tensor(_inputs(4, B), device=cuda).to(torch.bfloat16)
    t = np.zeros((B, mdg.MLP_OUT_PAD), np.float32)
    t[:, :mdg.MLP_OUT] = wl.uniform_range(-1, 1, 5, 12, 0, np.arange(B, dtype=np.uint64)[:, None],
                                          np.arange(mdg.MLP_OUT, dtype=np.uint64)[None, :])
    loss = torch.zeros(1, device=cuda)
    m.grad(x, torch.as_tensor(t, device=cuda), loss)
    torch.cuda.synchronize()
    g = mdg.mlp_unflatten(m.grads())
    # the oracle network with the 13 used outputs
    p13 = _f64(layers)
    p13[3] = (p13[3][0][:mdg.MLP_OUT], p13[3][1][:mdg.MLP_OUT])
    xo = x.float().cpu().numpy().astype(np.float64)
    yo, cache = omlp.forward(p13, xo, bf16_storage=True)
    go = omlp.backward(p13, cache, yo, t[:, :mdg.MLP_OUT].astype(np.float64), bf16_storage=True)
    assert float(loss) == pytest.approx(omlp.mse(yo, t[:, :mdg.MLP_OUT]), rel=1e-3)
    for l in range(4):
        gw, gb = g[l]
        if l == 3:
            assert np.all(gw[mdg.MLP_OUT:] == 0) and np.all(gb[mdg.MLP_OUT:] == 0)
            gw, gb = gw[:mdg.MLP_OUT], gb[:mdg.MLP_OUT]
        for a, b in ((gw, go[l][0]), (gb, go[l][1])):
            rel = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert rel < 2e-2, f"layer {l}: relative gradient error {rel:.3g}"
    assert np.all(g[0][0][:, mdg.MLP_IN:] == 0)  # padded inputs get no gradient


@pytest.mark.parametrize("B", [128, 384, 9856])
def test_gradients_over_uneven_tile_shares(cuda, B):
    """One tile, fewer tiles than shares, and 77 tiles in shares of 4 and 7 with the last ones
    short or empty: the bounds of the weight-gradient kernel's split over the batch."""
    test_gradients_and_loss_match_oracle(cuda, mdg.MLP_PATH_TCGEN05, B)


def test_weight_gradients_of_a_large_batch(cuda):
    """The output layer's gradients of 131072 rows, whose sums grow without cancelling, against the same
    network in float64 with the same bf16 roundings. Activations near a bf16 rounding boundary flip on one
    side (about 1e-4 of them, by 2^-8: 1e-7 over the batch); the tensor cores cut FP32 sums off by up to
    2^-24 every 16 rows, 48 times in a run, 3e-6; the additions of 171 runs round to 2^-24 each, 1e-6."""
    B = 131072
    layers = _layers(61)
    m = mdg.MLP(B, layers)
    g = torch.Generator(device=cuda)
    g.manual_seed(62)
    x = torch.zeros((B, mdg.MLP_IN_PAD), device=cuda)
    x[:, :mdg.MLP_IN] = torch.randn((B, mdg.MLP_IN), generator=g, device=cuda)
    x = x.bfloat16()
    t = torch.full((B, mdg.MLP_OUT_PAD), 4.0, device=cuda)
    m.grad(x, t)
    assert m.status() == 0
    W4, b4 = mdg.mlp_unflatten(m.grads())[3]
    h = x.double()
    for l in range(4):
        W, b = (torch.as_tensor(np.asarray(a, np.float32), device=cuda) for a in layers[l])
        z = h @ W.bfloat16().double().T + b.double()
        h = (z * torch.sigmoid(z)).float().bfloat16().double() if l < 3 else h
    d = (z - t.double()) * (torch.arange(mdg.MLP_OUT_PAD, device=cuda) < mdg.MLP_OUT)
    dy = (d * (2 / (B * mdg.MLP_OUT))).float().bfloat16().double()
    for got, want in ((W4, dy.T @ h), (b4, dy.sum(0))):
        got = torch.as_tensor(got, device=cuda).double()
        assert float((got - want).norm() / want.norm()) < 5e-6


@pytest.mark.parametrize("path", [mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_MMA_SYNC])
def test_silu_of_far_negative_pre_activations(cuda, path):
    """SiLU is a full division in training, up to where exp(-z) overflows: with z = -88 in the whole first
    layer h is -88 / (1 + e^88) = -5.3e-37, no zero, and the second layer's weight gradient is h times its
    bias gradient. Both round to bf16 once (2^-9) and sum 128 rows of one sign pattern in FP32."""
    B = 128
    layers = [(np.array(W, np.float32), np.array(b, np.float32)) for W, b in _layers(51)]
    layers[0][0][:], layers[0][1][:], layers[1][0][:] = 0.0, -88.0, 0.0
    m = mdg.MLP(B, layers)
    m.set_train_path(path)
    x = torch.as_tensor(_inputs(52, B), device=cuda).to(torch.bfloat16)
    t = torch.full((B, mdg.MLP_OUT_PAD), 1e10, device=cuda)
    m.grad(x, t)
    assert m.status() == 0
    g = mdg.mlp_unflatten(m.grads())
    h = -88.0 / (1.0 + np.exp(88.0))
    want = np.outer(g[1][1], np.full(mdg.MLP_HIDDEN, h))
    assert np.abs(want).max() > 1e-35
    np.testing.assert_allclose(g[1][0], want, rtol=2.0 ** -7, atol=2.0 ** -7 * np.abs(want).max())


@pytest.mark.parametrize("path", [mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_MMA_SYNC])
def test_loss_at_any_address(cuda, path):
    """The loss goes to any address that a copy can reach: one that is not 4-byte aligned (no kernel
    stores to it) receives the same four bytes, and its neighbours stay as they were."""
    B = 128
    m = mdg.MLP(B, _layers(31))
    m.set_train_path(path)
    x = torch.as_tensor(_inputs(32, B), device=cuda).to(torch.bfloat16)
    t = torch.full((B, mdg.MLP_OUT_PAD), 0.25, device=cuda)
    loss = torch.zeros(1, device=cuda)
    m.grad(x, t, loss)
    buf = torch.full((12,), 7, dtype=torch.uint8, device=cuda)
    stream = torch.cuda.current_stream().cuda_stream
    assert mdg.lib().mdg_mlp_grad(m._m, x.data_ptr(), t.data_ptr(), B, buf.data_ptr() + 5, stream) == mdg.OK
    got = buf.cpu().numpy()
    # mma.sync adds its partial losses up with atomics, in any order
    np.testing.assert_allclose(got[5:9].view(np.float32), loss.cpu().numpy(), rtol=0 if path == mdg.MLP_PATH_TCGEN05 else 1e-6)
    assert float(loss) > 0 and np.all(np.delete(got, slice(5, 9)) == 7)


def test_adam_refreshes_the_weight_image(cuda):
    """The forward pass after an Adam step equals, bit for bit, that of a network created with
    the updated parameters (whose image is built from their bf16 copies)."""
    B = 256
    m = mdg.MLP(B, _layers(21))
    x = torch.as_tensor(_inputs(22, B), device=cuda).to(torch.bfloat16)
    t = torch.full((B, mdg.MLP_OUT_PAD), 0.25, device=cuda)
    for _ in range(2):
        m.grad(x, t)
        m.adam(1e-2)
    fresh = mdg.MLP(B, m.params())
    for path in (mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_TCGEN05_PAIRS):
        ys = []
        for net in (m, fresh):
            net.set_path(path)
            y = torch.empty((B, mdg.MLP_OUT_PAD), device=cuda)
            net.forward(x, y)
            ys.append(y)
        assert torch.equal(*ys)


@pytest.mark.parametrize("path", [mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_TCGEN05_PAIRS])
def test_weights_around_captured_calls(cuda, path):
    """Calls that were captured and have not run change nothing: the forward pass after a captured,
    unplayed training step equals that of another network with the same parameters, bit for bit. And
    a captured forward pass reads the parameters set after its capture."""
    B = 256
    x = torch.as_tensor(_inputs(42, B), device=cuda).to(torch.bfloat16)
    t = torch.full((B, mdg.MLP_OUT_PAD), 0.25, device=cuda)

    def forward(net):
        y = torch.empty((B, mdg.MLP_OUT_PAD), device=cuda)
        net.forward(x, y)
        return y
    nets = [mdg.MLP(B, _layers(41)), mdg.MLP(B, _layers(41)), mdg.MLP(B, _layers(43))]
    for net in nets:
        net.set_path(path)
    want = [forward(net) for net in nets[1:]]
    m = nets[0]
    train, infer = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    loss = torch.zeros(1, device=cuda)
    with torch.cuda.graph(train):
        m.grad(x, t, loss)
        m.adam(1e-2)
    assert torch.equal(forward(m), want[0])
    y = torch.zeros((B, mdg.MLP_OUT_PAD), device=cuda)
    with torch.cuda.graph(infer):
        m.forward(x, y)
    m.set_params(nets[2].params())
    infer.replay()
    assert torch.equal(y, want[1])
    train.replay()
    assert not torch.equal(forward(m), want[1]) and float(loss) > 0


def test_adam_matches_oracle(cuda):
    B = 128
    layers = _layers(6)
    m = mdg.MLP(B, layers)
    x = torch.as_tensor(_inputs(7, B), device=cuda).to(torch.bfloat16)
    t = torch.zeros((B, mdg.MLP_OUT_PAD), device=cuda)
    t[:, :mdg.MLP_OUT] = 0.5
    params = _f64(mdg.mlp_unflatten(m.params()))
    mo, vo = omlp.adam_init(params)
    for step in (1, 2, 3):
        m.grad(x, t)
        torch.cuda.synchronize()
        grads = _f64(mdg.mlp_unflatten(m.grads()))
        m.adam(1e-3)
        torch.cuda.synchronize()
        params, mo, vo = omlp.adam_step(params, grads, mo, vo, step, lr=1e-3)
        got = mdg.mlp_unflatten(m.params())
        for (Wg, bg), (Wo, bo) in zip(got, params):
            np.testing.assert_allclose(Wg, Wo, rtol=1e-5, atol=1e-7)
            np.testing.assert_allclose(bg, bo, rtol=1e-5, atol=1e-7)


def test_training_reduces_the_loss(cuda):
    B, rows = 512, 4096
    teacher = _f64(_layers(8, bias_scale=0.5))
    teacher[3] = (teacher[3][0][:mdg.MLP_OUT] * 0.3, teacher[3][1][:mdg.MLP_OUT])
    xn = _inputs(9, rows)
    yt, _ = omlp.forward(teacher, xn.astype(np.float64))
    t = np.zeros((rows, mdg.MLP_OUT_PAD), np.float32)
    t[:, :mdg.MLP_OUT] = (yt - yt.mean(0)) / yt.std(0)
    m = mdg.MLP(B, wl.mlp_init(10))
    x = torch.as_tensor(xn, device=cuda).to(torch.bfloat16)
    tt = torch.as_tensor(t, device=cuda)
    loss = torch.zeros(1, device=cuda)
    first = None
    for it in range(400):
        sl = slice((it % (rows // B)) * B, (it % (rows // B) + 1) * B)
        m.grad(x[sl].contiguous(), tt[sl].contiguous(), loss)
        if first is None:
            first = float(loss)
        m.adam(2e-3)
    torch.cuda.synchronize()
    assert float(loss) < 0.1 * first


def test_features_match_state_and_oracle_neighbours(cuda):
    sw = wl.full_aero(13, n_envs=150)
    h = mdg.Handle(sw.drones_per_env, sw.flags)
    state = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
    rpm = torch.as_tensor(wl.rpm_actions(13, sw.n, 0, HOVER), device=cuda)
    raw = torch.empty((sw.n, mdg.MLP_IN), device=cuda)
    h.features(state, rpm, raw)
    torch.cuda.synchronize()
    raw = raw.cpu().numpy()
    x, _, _ = oracle_arrays(state)
    np.testing.assert_array_equal(raw[:, :13], x.astype(np.float32))
    np.testing.assert_array_equal(raw[:, 13:17], rpm.cpu().numpy())
    env_off = sw.env_off
    for e in range(sw.n_envs):
        b, N = int(env_off[e]), int(sw.drones_per_env[e])
        xe = x[b:b + N]
        for j in range(N):
            # the drone each listed slot describes (the one whose relative position it holds),
            # then that list checked as a valid 4-nearest list and the features against it
            listed = np.full(4, -1)
            for k in range(min(4, N - 1)):
                dp = np.abs(xe[:, 0:3] - xe[j, 0:3] - raw[b + j, 17 + 6 * k:20 + 6 * k]).sum(axis=1)
                dp[j] = np.inf
                listed[k] = b + int(np.argmin(dp))
            r_ref, _ = assert_knn_valid(xe, j, b, listed, what=f"features of drone {b + j}")
            assert excess(raw[b + j, 17:], r_ref, 1e-6, floor=1e-2) <= 1.0


@pytest.fixture(scope="module")
def trained(cuda):
    raw, delta = sg.generate_transitions(4096, 24, seed=21, device=cuda)
    data = sg.Dataset(raw, delta)
    m = mdg.MLP(8192, wl.mlp_init(22))
    data.attach(m)
    hist = sg.fit(m, data, epochs=6, batch=8192, lr=2e-3)
    return m, data, hist


def test_surrogate_step_gains_over_no_network(cuda, trained):
    m, data, hist = trained
    assert hist[-1] < 0.5 * hist[0]
    sw = wl.full_aero(77, n_envs=1024)
    h = mdg.Handle(sw.drones_per_env, sw.flags)
    s_sur = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
    s_pln = s_sur.clone()
    before = sg.state13(s_sur).clone()
    wp = torch.as_tensor(wl.waypoints(77, sw.n), device=cuda)
    nfb = torch.zeros(1, dtype=torch.int32, device=cuda)
    m.step(h, s_sur, wp, mdg.ACT_PID, 5, 4.0, nfb)
    h.step(s_pln, wp, mdg.ACT_PID, 5)
    torch.cuda.synchronize()
    xs, xp = sg.state13(s_sur), sg.state13(s_pln)
    true_d = xp - before
    n_fb = int(nfb)
    assert n_fb < 0.5 * sw.n_envs
    # Evaluate where the network is meant to work: drones not sent to the integrator whose
    # true state change lies in the regular regime the network was trained on (standardised
    # change within +-8); the rest is the chaotic tail of near-coincident heights.
    zt = (true_d - data.out_mean) / data.out_std
    diff = (xs - xp).abs().max(dim=1).values
    env_fb = (diff.view(-1, 4) == 0).all(dim=1).repeat_interleave(4)  # fallback envs match the plain step
    regular = (zt.abs() <= 8).all(dim=1) & ~env_fb
    assert float(regular.float().mean()) > 0.5
    # One-step error of the surrogate vs the plain integrator against the error of a
    # predictor without the network (state unchanged). The rotational change depends on
    # the motor torques alone and is learned closely (this small training: 0.22 quaternion,
    # 0.085 body rate). The translational change is dominated by the downwash law's 1/dz^2:
    # the formation's drones fly at nearly equal heights (median 1.1 cm to the nearest other
    # height), which the network does not represent; velocity is required to gain (0.955
    # measured), position only not to lose more than 10% (1.06 measured: the network's
    # spurious vertical motion costs about what it gains).
    for name, sl, bound in (("quaternion", slice(3, 7), 0.3), ("body rate", slice(10, 13), 0.3),
                            ("position", slice(0, 3), 1.1), ("velocity", slice(7, 10), 1.0)):
        err = (xs[regular, sl] - xp[regular, sl]).pow(2).mean().sqrt()
        base = true_d[regular, sl].pow(2).mean().sqrt()
        assert err < bound * base, f"{name}: surrogate rms error {float(err):.3g} vs no-network {float(base):.3g}"
    # quaternions stay unit
    q = xs[:, 3:7]
    assert torch.allclose(q.norm(dim=1), torch.ones_like(q[:, 0]), atol=1e-5)


def test_out_of_distribution_environments_take_the_integrator(cuda, trained):
    m, data, _ = trained
    sw = wl.full_aero(78, n_envs=300)
    h = mdg.Handle(sw.drones_per_env, sw.flags)
    state = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
    x0, i0, a0 = oracle_arrays(state)
    wp = wl.waypoints(78, sw.n)
    nfb = torch.zeros(1, dtype=torch.int32, device=cuda)
    m.step(h, state, torch.as_tensor(wp, device=cuda), mdg.ACT_PID, 5, 0.0, nfb)  # everything out of distribution
    torch.cuda.synchronize()
    assert int(nfb) == sw.n_envs
    xg, ig, _ = oracle_arrays(state)
    layout = (sw.drones_per_env, sw.flags)
    acts = np.full(sw.n_envs, mdg.ACT_PID)
    xo, io, _ = oracle_step(P, layout, x0, i0, a0, wp, acts, 5)
    resp = tolerance_response(P, layout, x0, i0, a0, wp, acts, 5)
    assert_horizon_close(xg, xo, resp, 5, what="fallback")
    assert excess(ig, io, 1e-5) <= 1.0
    assert h.status()[0] == mdg.OK


@pytest.mark.parametrize("integrator", ["euler", "rk4"])
def test_fallback_of_large_environments(cuda, trained, integrator):
    """Environments of 64 drones (the dense swarm's size, one block per environment in the
    fallback) and Runge-Kutta substeps: with every environment out of distribution the
    surrogate step is the plain integrator, against the oracle over the control step (heights
    spread per environment, so that the downwash is well conditioned)."""
    m, data, _ = trained
    sw = spread_heights(wl.dense(80, n_envs=24), dz=0.3, z0=0.5)
    c = mdg.Constants.cf2x()
    Po = oracle.cf2x()
    if integrator == "rk4":
        c.integrator = mdg.INTEGRATOR_RK4
        Po.integrator = oracle.RK4
    h = mdg.Handle(sw.drones_per_env, sw.flags, c)
    state = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
    x0, i0, a0 = oracle_arrays(state)
    act = wl.rpm_actions(80, sw.n, 0, HOVER)
    nfb = torch.zeros(1, dtype=torch.int32, device=cuda)
    m.step(h, state, torch.as_tensor(act, device=cuda), mdg.ACT_RPM, 5, 0.0, nfb)
    torch.cuda.synchronize()
    assert int(nfb) == sw.n_envs
    xg, _, ag = oracle_arrays(state)
    layout = (sw.drones_per_env, sw.flags)
    acts = np.full(sw.n_envs, mdg.ACT_RPM)
    xo, _, ao = oracle_step(Po, layout, x0, i0, a0, act, acts, 5)
    resp = tolerance_response(Po, layout, x0, i0, a0, act, acts, 5)
    assert_horizon_close(xg, xo, resp, 5, what=f"fallback of 64-drone environments ({integrator})")
    np.testing.assert_allclose(ag, ao, rtol=1e-6)
    assert h.status()[0] == mdg.OK


def test_surrogate_step_paths_agree(cuda, trained):
    m, data, _ = trained
    sw = wl.full_aero(79, n_envs=512)
    h = mdg.Handle(sw.drones_per_env, sw.flags)
    wp = torch.as_tensor(wl.waypoints(79, sw.n), device=cuda)
    out = []
    for path in (mdg.MLP_PATH_MMA_SYNC, mdg.MLP_PATH_TCGEN05, mdg.MLP_PATH_TCGEN05_PAIRS):
        m.set_path(path)
        st = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
        m.step(h, st, wp, mdg.ACT_PID, 5, 4.0)
        torch.cuda.synchronize()
        out.append(sg.state13(st).cpu().numpy().astype(np.float64))
    m.set_path(mdg.MLP_PATH_TCGEN05_PAIRS)  # the default
    # same network, same inputs and the same out-of-distribution decisions: the states differ
    # only by out_std times the difference of the standardised outputs, which the forward
    # test bounds by 1e-2 max(|y|, 1); |y| stays below ~4 in distribution, hence 0.05 out_std
    tol = 0.05 * data.out_std.cpu().numpy().astype(np.float64)
    for o in out[1:]:
        assert np.all(np.abs(o - out[0]) <= tol[None, :])
    assert h.status()[0] == mdg.OK


def test_transition_is_features_then_step(cuda):
    """mdg_transition: the applied RPMs are rpm times rpm_scale, the inputs are mdg_features of
    the state with them, the state advances by mdg_step, and delta is after minus before."""
    sw = wl.full_aero(14, n_envs=200)
    h = mdg.Handle(sw.drones_per_env, sw.flags)
    s_a = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
    s_b = s_a.clone()
    rpm = torch.as_tensor(wl.rpm_actions(14, sw.n, 0, HOVER), device=cuda)
    scale = torch.as_tensor(wl.uniform_range(0.9, 1.1, 14, 13, 0, np.arange(sw.n, dtype=np.uint64)[:, None],
                                             np.arange(4, dtype=np.uint64)[None, :]), device=cuda)
    applied = torch.empty_like(rpm)
    raw = torch.empty((sw.n, mdg.MLP_IN), device=cuda)
    delta = torch.empty((sw.n, mdg.MLP_OUT), device=cuda)
    h.transition(s_a, rpm, applied, raw, delta, rpm_scale=scale)
    ref_rpm = rpm * scale
    raw_b = torch.empty_like(raw)
    before = sg.state13(s_b).clone()
    h.features(s_b, ref_rpm, raw_b)
    h.step(s_b, ref_rpm, mdg.ACT_RPM, 5)
    torch.cuda.synchronize()
    assert torch.equal(applied, ref_rpm)
    assert torch.equal(raw, raw_b) and torch.equal(s_a, s_b)
    assert torch.equal(delta, sg.state13(s_b) - before)


def test_fit_normalization_matches_its_definition(cuda):
    """mdg_mlp_fit_normalization against the same steps in numpy (float64): non-finite rows
    dropped; per column the 0.5% / 99.5% quantiles (linear interpolation) of an evenly strided
    sample, widened by 10% of their distance, as the trim box; FP64 mean and unbiased standard
    deviation of the kept rows (scale 1 for a constant column); rows with a standardised input
    beyond +-4 or target beyond +-8 dropped; the kept inputs' range widened by 10% plus 1e-6 as
    the out-of-distribution box; the standardised rows in order, truncated to a multiple of 128."""
    rng = np.random.default_rng(5)
    N = 300_000  # above the 262144-row sample: stride 1 (the stride is 2 only from 524288 rows)
    raw = rng.standard_normal((N, mdg.MLP_IN)).astype(np.float32) * np.linspace(0.1, 3, mdg.MLP_IN)[None, :].astype(np.float32)
    delta = rng.standard_normal((N, mdg.MLP_OUT)).astype(np.float32)
    raw[:, 5] = 2.5  # a constant column
    heavy = rng.random(N) < 0.01  # a heavy tail the trim removes
    delta[heavy, 3] *= 1e3
    raw[rng.integers(0, N, 50), 7] = np.nan
    delta[rng.integers(0, N, 50), 2] = np.inf
    m = mdg.MLP(128)
    x = torch.empty((N, mdg.MLP_IN_PAD), dtype=torch.bfloat16, device=cuda)
    t = torch.empty((N, mdg.MLP_OUT_PAD), device=cuda)
    n_fin, n_kept = m.fit_normalization(torch.as_tensor(raw, device=cuda), torch.as_tensor(delta, device=cuda), x, t)
    in_mean, in_std, out_mean, out_std, in_lo, in_hi = m.normalization()
    # the definition, in numpy
    A = np.concatenate([raw, delta], 1).astype(np.float64)
    fin = np.isfinite(A).all(1)
    F = A[fin]
    assert n_fin == F.shape[0]
    stride = max(1, F.shape[0] // 262144)
    S = F[::stride]
    qlo, qhi = np.quantile(S, 0.005, axis=0), np.quantile(S, 0.995, axis=0)
    r = qhi - qlo
    keep1 = ((F >= qlo - 0.1 * r) & (F <= qhi + 0.1 * r)).all(1)
    K1 = F[keep1]
    mean = K1.mean(0)
    sd = K1.std(0, ddof=1)
    sd = np.where(sd > 1e-6 * np.maximum(np.abs(mean), 1.0), sd, 1.0)
    np.testing.assert_allclose(in_mean, mean[:mdg.MLP_IN], rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(out_mean, mean[mdg.MLP_IN:], rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(in_std, sd[:mdg.MLP_IN], rtol=1e-5)
    np.testing.assert_allclose(out_std, sd[mdg.MLP_IN:], rtol=1e-5)
    assert in_std[5] == 1.0
    Z = (K1 - mean) / sd
    keep2 = (np.abs(Z[:, :mdg.MLP_IN]) <= 4.0).all(1) & (np.abs(Z[:, mdg.MLP_IN:]) <= 8.0).all(1)
    K2 = K1[keep2]
    assert abs(K2.shape[0] // 128 * 128 - n_kept) <= 128  # boundary rows may round either way in float32
    lo, hi = K2[:, :mdg.MLP_IN].min(0), K2[:, :mdg.MLP_IN].max(0)
    pad = 0.1 * (hi - lo) + 1e-6
    np.testing.assert_allclose(in_lo, lo - pad, rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(in_hi, hi + pad, rtol=1e-5, atol=1e-5)
    # the emitted rows: the kept rows in order, standardised
    xs = x[:n_kept].float().cpu().numpy()
    ts = t[:n_kept].cpu().numpy()
    n_cmp = min(n_kept, K2.shape[0]) // 2  # rows before any boundary difference
    zin = (K2[:n_cmp, :mdg.MLP_IN] - mean[:mdg.MLP_IN]) / sd[:mdg.MLP_IN]
    np.testing.assert_allclose(xs[:n_cmp, :mdg.MLP_IN], zin, rtol=1e-2, atol=1e-2)
    assert np.all(xs[:, mdg.MLP_IN:] == 0) and np.all(ts[:, mdg.MLP_OUT:] == 0)
    np.testing.assert_allclose(ts[:n_cmp, :mdg.MLP_OUT], Z[keep2][:n_cmp, mdg.MLP_IN:], rtol=1e-4, atol=1e-4)


@pytest.mark.parametrize("recipe", ["full_aero", "full_aero_ragged", "dense", "dense_pid"])
def test_surrogate_step_composes_its_parts(cuda, trained, recipe):
    """mdg_surrogate_step equals its parts called one by one: the plain integrator's inputs of
    the state and its RPMs (mdg_transition), their standardisation (mdg_mlp_standardize), the
    network (mdg_mlp_forward) and the de-standardised change added on the host (quaternion
    renormalised), on 4-drone (PID; also a drone count that is not a multiple of 128) and
    64-drone (RPM and PID) environments. With the trained box every
    environment with an input outside it is counted for the fallback; with an unbounded box
    none is, and every drone is compared."""
    _, data, _ = trained
    # full_aero_ragged: 1204 drones, not a multiple of the network's 128-row tiles: the last
    # tile holds padding rows, which the fused update must not write (a row past the end of a
    # state plane is the next plane's first drone, compared below)
    sw = (wl.full_aero(81, n_envs=256) if recipe == "full_aero" else
          wl.full_aero(83, n_envs=301) if recipe == "full_aero_ragged" else wl.dense(82, n_envs=16))
    h = mdg.Handle(sw.drones_per_env, sw.flags)
    if recipe == "dense":
        action, act = torch.as_tensor(wl.rpm_actions(82, sw.n, 0, HOVER), device=cuda), mdg.ACT_RPM
    else:
        action, act = torch.as_tensor(wl.waypoints(81, sw.n), device=cuda), mdg.ACT_PID
    in_mean, in_std, out_mean, out_std, in_lo, in_hi = data.stats()
    for bounded in (True, False):
        m = mdg.MLP((sw.n + 127) // 128 * 128, wl.mlp_init(23))
        lo, hi = (in_lo, in_hi) if bounded else (np.full_like(in_lo, -1e30), np.full_like(in_hi, 1e30))
        m.set_normalization(in_mean, in_std, out_mean, out_std, lo, hi)
        ood_z = 4.0 if bounded else 1e30
        state = mdg.pack_state(sw.p, sw.q, sw.v, sw.w, device=cuda)
        before = state.clone()
        nfb = torch.zeros(1, dtype=torch.int32, device=cuda)
        m.step(h, state, action, act, 5, ood_z, nfb)
        # the parts: RPMs (the PID on a copy of the state), inputs, standardisation, network
        s2 = before.clone()
        rpm = torch.empty((sw.n, 4), device=cuda)
        if act == mdg.ACT_PID:
            h.pid(s2, action, rpm)
        else:
            rpm.copy_(action.clamp(0.0, mdg.Constants.cf2x().max_rpm()))
        raw = torch.empty((sw.n, mdg.MLP_IN), device=cuda)
        delta = torch.empty((sw.n, mdg.MLP_OUT), device=cuda)
        applied = torch.empty((sw.n, 4), device=cuda)
        h.transition(s2.clone(), rpm, applied, raw, delta)
        rows = (sw.n + 127) // 128 * 128
        x = torch.zeros((rows, mdg.MLP_IN_PAD), dtype=torch.bfloat16, device=cuda)
        m.standardize(raw, x[:sw.n])
        y = torch.empty((rows, mdg.MLP_OUT_PAD), device=cuda)
        m.forward(x, y)
        torch.cuda.synchronize()
        rawn = raw.cpu().numpy().astype(np.float64)
        z = (rawn - in_mean) / in_std
        bad = ~((np.abs(z) <= ood_z) & (rawn >= lo) & (rawn <= hi))
        env_bad = bad.reshape(sw.n_envs, -1).any(axis=1)
        assert int(nfb) == int(env_bad.sum()), (int(nfb), int(env_bad.sum()))
        if bounded:
            continue
        assert int(nfb) == 0
        d = y[:sw.n, :mdg.MLP_OUT].double().cpu().numpy() * out_std + out_mean
        x0 = sg.state13(before).double().cpu().numpy()
        want = x0 + d
        want[:, 3:7] /= np.linalg.norm(want[:, 3:7], axis=1, keepdims=True)
        got = sg.state13(state).double().cpu().numpy()
        assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(np.abs(want), 1.0)), np.abs(got - want).max()


@pytest.mark.parametrize("sizes,block", [([1] * 33, None), ([3, 1, 5, 2, 33], None), ([64] * 3, None), ([7] * 11, 1024),
                                         ([1000, 24], None)])
def test_transition_rows_at_warp_edges(cuda, sizes, block):
    """The staged rows of partial warps, uneven tiles and the largest block: the inputs are the
    state's and the RPMs' own values, the change is the difference of the states, exactly, and
    nothing beyond the rows is written."""
    dpe = np.array(sizes, np.int32)
    n = int(dpe.sum())
    p, q, v, w = wl.random_states(501, n, pos_scale=3.0, z0=4.0)
    h = mdg.Handle(dpe, np.full(len(dpe), 3, np.uint32))
    if block:
        h.set_block_size(block)
    s0 = mdg.pack_state(p, q, v, w, device=cuda)
    s1 = s0.clone()
    rpm = torch.as_tensor(wl.rpm_actions(502, n, 0, 14468.0), device=cuda)
    scale = torch.as_tensor(wl.uniform_range(0.9, 1.1, 503, 12, 0, np.arange(n, dtype=np.uint64)[:, None],
                                             np.arange(4, dtype=np.uint64)[None, :]), device=cuda)
    applied = torch.empty((n, 4), device=cuda)
    buf = [torch.full((n * m + 64,), 7.0, device=cuda) for m in (mdg.MLP_IN, mdg.MLP_OUT)]
    raw, delta = (b[:n * m].reshape(n, m) for b, m in zip(buf, (mdg.MLP_IN, mdg.MLP_OUT)))
    h.transition(s1, rpm, applied, raw, delta, rpm_scale=scale)
    assert torch.equal(applied, rpm * scale)
    assert torch.equal(raw[:, :13], sg.state13(s0)) and torch.equal(raw[:, 13:17], applied)
    assert torch.equal(delta, sg.state13(s1) - sg.state13(s0))
    _, idx, rel = h.new_obs(cuda)
    kin = torch.empty((n, mdg.KIN_DIM), device=cuda)
    h.obs(s0, kin, idx, rel)
    assert torch.equal(raw[:, 17:], rel)
    assert all(torch.all(b[n * m:] == 7.0) for b, m in zip(buf, (mdg.MLP_IN, mdg.MLP_OUT)))


@pytest.mark.parametrize("N", [130, 1024, 1025, 40003, 600001])
def test_fit_normalization_at_tile_edges(cuda, N):
    """Row counts around the tiles' sizes and, at 600001, a sample stride of 2: statistics and rows
    against numpy in float64, and the same result, bit for bit, from sets that are only 4-byte
    aligned (the scalar copies). Tolerances: the statistics round to float32 once (6e-8; 1e-6 allows
    the box edges' own rounding to move no row), targets take one subtraction and one division
    (2e-7 of the largest term, at most 8 standard deviations about a mean of at most 2)."""
    rng = np.random.default_rng(N)
    raw = (rng.standard_normal((N, mdg.MLP_IN)) * np.linspace(0.1, 3, mdg.MLP_IN) + 2.0).astype(np.float32)
    delta = rng.standard_normal((N, mdg.MLP_OUT)).astype(np.float32)
    raw[:, 40] = 0.0
    raw[N // 2, 3] = np.inf
    delta[N - 1, 12] = np.nan
    got = []
    for shift in (0, 1):  # floats in front of each set
        buf = [torch.zeros(a.size + shift, device=cuda) for a in (raw, delta)]
        sets = []
        for b, a in zip(buf, (raw, delta)):
            b[shift:] = torch.as_tensor(a.reshape(-1), device=cuda)
            sets.append(b[shift:].reshape(a.shape))
        m = mdg.MLP(128)
        x = torch.zeros((N, mdg.MLP_IN_PAD), dtype=torch.bfloat16, device=cuda)
        t = torch.zeros((N, mdg.MLP_OUT_PAD), device=cuda)
        got.append((m.fit_normalization(*sets, x, t), m.normalization(), x, t))
    (counts, norm, x, t), (counts1, norm1, x1, t1) = got
    assert counts == counts1 and all(np.array_equal(a, b) for a, b in zip(norm, norm1))
    assert torch.equal(x, x1) and torch.equal(t, t1)
    F = np.concatenate([raw, delta], 1).astype(np.float64)
    F = F[np.isfinite(F).all(1)]
    assert counts[0] == N - 2 == F.shape[0]
    S = F[::max(1, F.shape[0] // 262144)]
    qlo, qhi = np.quantile(S, float(np.float32(0.005)), axis=0), np.quantile(S, 1 - float(np.float32(0.005)), axis=0)
    lo, hi = (qlo - 0.1 * (qhi - qlo)).astype(np.float32), (qhi + 0.1 * (qhi - qlo)).astype(np.float32)
    K = F[((F >= lo) & (F <= hi)).all(1)]
    mean, sd = K.mean(0), K.std(0, ddof=1)
    sd[40] = 1.0
    np.testing.assert_allclose(np.concatenate([norm[0], norm[2]]), mean, rtol=1e-6, atol=1e-7)
    np.testing.assert_allclose(np.concatenate([norm[1], norm[3]]), sd, rtol=1e-6)
    Z = (K - mean) / sd
    Z = Z[(np.abs(Z[:, :mdg.MLP_IN]) <= 4.0).all(1) & (np.abs(Z[:, mdg.MLP_IN:]) <= 8.0).all(1)]
    n = Z.shape[0] // 128 * 128
    assert counts[1] == n
    np.testing.assert_allclose(t[:n, :mdg.MLP_OUT].cpu().numpy(), Z[:n, mdg.MLP_IN:], rtol=1e-6, atol=3e-6)
    # bf16: half an ulp (2^-9 relative) of the float32 value
    np.testing.assert_allclose(x[:n, :mdg.MLP_IN].float().cpu().numpy(), Z[:n, :mdg.MLP_IN], rtol=2.0 ** -8, atol=1e-4)
    assert not x[:n, mdg.MLP_IN:].any() and not t[:n, mdg.MLP_OUT:].any() and not x[n:].any() and not t[n:].any()


@pytest.mark.parametrize("margin", [0.0, 1e6, 1e12, 3e30, np.inf])
def test_fit_normalization_statistics_at_any_margin(cuda, margin):
    """Mean and deviation are taken in float64 about the mean itself, whatever the box: with wide margins
    (a caller that does not trim), with columns far from zero against their spread, with one far row, with
    tiny and with huge columns (the largest margins overflow, so that their limits are infinite; an infinite
    one leaves no limit to a constant column, so none is kept). They round to float32 once (6e-8; the
    float64 sums are good to 1e-13 of the far row's square, 1e-9 of the variance here)."""
    N = 30007
    rng = np.random.default_rng(7)
    F = rng.standard_normal((N, mdg.MLP_IN + mdg.MLP_OUT))
    F[:, 0] += 1e4
    F[:, 1] = 1e4 + 0.05 * F[:, 1]
    F[:, 2] *= 1e-20
    F[:, 3] *= 1e25
    F[N // 2, 4] = 1e3
    F[:, 6] = 5e-42 + 1e-42 * F[:, 6]
    F[:, 7] = 3e38 * (F[:, 7] > 0) - 1e38
    if np.isfinite(margin):
        F[:, 5] = 0.1
    F = F.astype(np.float32)
    raw, delta = F[:, :mdg.MLP_IN].copy(), F[:, mdg.MLP_IN:].copy()
    m = mdg.MLP(128)
    x = torch.zeros((N, mdg.MLP_IN_PAD), dtype=torch.bfloat16, device=cuda)
    t = torch.zeros((N, mdg.MLP_OUT_PAD), device=cuda)
    big = 3e38
    counts = m.fit_normalization(torch.as_tensor(raw, device=cuda), torch.as_tensor(delta, device=cuda), x, t, trim_frac=0.0,
                                 margin=margin, ood_z=big, target_clip=big)
    assert counts == (N, N // 128 * 128)  # the quantiles 0 and 1 keep every row
    K = F.astype(np.float64)
    mean, sd = K.mean(0), K.std(0, ddof=1)
    sd = np.where(sd > 1e-6 * np.maximum(np.abs(mean), 1.0), sd, 1.0)
    norm = m.normalization()
    scale = np.maximum(np.abs(mean), np.abs(K).mean(0) * 1e-6)
    assert np.all(np.abs(np.concatenate([norm[0], norm[2]]) - mean) <= 1.2e-7 * scale + 1.4e-45)
    np.testing.assert_allclose(np.concatenate([norm[1], norm[3]]), sd, rtol=2e-7)


def _fit_digest(cuda):
    """Digest of what fit_normalization returns for a set below and one above the sample's first stride."""
    digest = hashlib.sha256()
    for N in (5003, 600001):
        g = torch.Generator(device=cuda)
        g.manual_seed(N)
        F = torch.randn((N, mdg.MLP_IN + mdg.MLP_OUT), generator=g, device=cuda)
        m = mdg.MLP(128)
        x = torch.zeros((N, mdg.MLP_IN_PAD), dtype=torch.bfloat16, device=cuda)
        t = torch.zeros((N, mdg.MLP_OUT_PAD), device=cuda)
        counts = m.fit_normalization(F[:, :mdg.MLP_IN].contiguous(), F[:, mdg.MLP_IN:].contiguous(), x, t)
        for a in (np.array(counts), *m.normalization(), x.view(torch.int16).cpu().numpy(), t.cpu().numpy()):
            digest.update(np.ascontiguousarray(a).tobytes())
    return digest.hexdigest()


def test_fit_normalization_with_a_small_workspace(cuda):
    """Where the sample of all columns finds no room it is taken a few columns at a time, with the same
    result bit for bit. The debug build takes the first workspace as refused."""
    from paper_2606_08039_gb300 import build
    build.build_library(debug=True)
    code = ("import sys; sys.path.insert(0, 'tests'); import torch; import test_gpu_surrogate as t; "
            "assert t.mdg.LIB_PATH.endswith('libmdg_debug.so'); print('digest', t._fit_digest(torch.device('cuda', 0)))")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, MDG_DEBUG_LIBRARY="1", PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    assert r.stdout.split()[-1] == _fit_digest(cuda)


def test_fit_normalization_without_usable_rows(cuda):
    """No finite row, and a single one: refused, and the outputs stay as they were."""
    m = mdg.MLP(128)
    for finite in (0, 1):
        raw = torch.full((300, mdg.MLP_IN), float("nan"), device=cuda)
        delta = torch.zeros((300, mdg.MLP_OUT), device=cuda)
        raw[:finite] = 1.0
        x = torch.ones((300, mdg.MLP_IN_PAD), dtype=torch.bfloat16, device=cuda)
        t = torch.ones((300, mdg.MLP_OUT_PAD), device=cuda)
        with pytest.raises(mdg.MdgError):
            m.fit_normalization(raw, delta, x, t)
        assert torch.all(x == 1) and torch.all(t == 1)


@pytest.mark.parametrize("size,envs,block", [(1, 300, None), (3, 43, None), (4, 33, 32), (7, 150, 1024), (33, 9, None),
                                             (1000, 3, None)])
def test_fallback_flags_at_tile_edges(cuda, size, envs, block):
    """Environments over uneven tiles and blocks, every third with one drone (another place in each)
    outside the box: exactly those take the integrator and are counted, also when the flags of an
    earlier step are still in the workspace; the others change by the network's prediction, here
    scaled to nothing, so their states stay as they were, exactly."""
    n = size * envs
    p, q, v, w = wl.random_states(511, n, pos_scale=3.0, z0=4.0)
    bad = np.arange(envs) % 3 == 0
    out = p.copy()
    out[(np.arange(envs) * size + np.arange(envs) % size)[bad], 2] = 200.0
    h = mdg.Handle(np.full(envs, size, np.int32), np.zeros(envs, np.uint32))
    if block:
        h.set_block_size(block)
    m = mdg.MLP((n + 127) // 128 * 128, _layers(4))
    lo, hi = np.full(mdg.MLP_IN, -1e30), np.full(mdg.MLP_IN, 1e30)
    hi[2] = 100.0
    m.set_normalization(np.zeros(mdg.MLP_IN), np.ones(mdg.MLP_IN), np.zeros(mdg.MLP_OUT), np.full(mdg.MLP_OUT, 1e-30), lo, hi)
    rpm = torch.zeros((n, 4), device=cuda)  # free fall
    nfb = torch.full((1,), -1, dtype=torch.int32, device=cuda)
    for pos, flagged in ((out, bad), (p, np.zeros(envs, bool)), (out, bad)):
        s0 = mdg.pack_state(pos, q, v, w, device=cuda)
        s1 = s0.clone()
        m.step(h, s1, rpm, mdg.ACT_RPM, 5, 1e30, nfb)
        assert int(nfb) == flagged.sum()
        a, b = (sg.state13(s).view(envs, size, 13)[:, :, [0, 1, 2, 7, 8, 9, 10, 11, 12]] for s in (s0, s1))
        same = (a == b).all(dim=2)
        f = torch.as_tensor(flagged, device=cuda)
        assert torch.all(same[~f]) and not torch.any(same[f])
    assert m.status() == 0 and h.status()[0] == mdg.OK
