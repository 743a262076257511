"""The FP32 layers on the tensor cores (operands split into bf16 parts): every channel combination, ragged images and
tiles, against the oracle's correlations, to the rounding of FP32 sums."""
import numpy as np
import pytest

from oracle import convnet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin", [2, 4, 32])
@pytest.mark.parametrize("cout", [2, 4, 32])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 16, 16), (1, 17, 15), (2, 50, 33)])
def test_forward_and_gradients_vs_oracle(cin, cout, shape):
    """Sums of n products rounded to FP32 stay within 4e-7 sqrt(n) of the largest result (an FMA chain's random walk, the
    bound the CUDA-core layers were held to); inputs over several decades."""
    import torch

    from paper_2407_05568_gb300 import es
    B, H, W = shape
    rng = np.random.default_rng(11 + 100 * cin + cout + H)
    a = (rng.standard_normal((B, cin, H, W)) * 10.0 ** rng.uniform(-2, 1, (B, cin, 1, 1))).astype(np.float32)
    w = convnet.bf16_round((rng.standard_normal((cout, cin, 3, 3)) / np.sqrt(9 * cin)).astype(np.float32))
    wt = torch.tensor(w, dtype=torch.bfloat16, device="cuda")
    b = rng.standard_normal(cout).astype(np.float32)
    at = torch.tensor(a, device="cuda")
    ws = torch.empty(es.es_nn_workspace_bytes(B, cin, cout, H, W) // 4 + 1, dtype=torch.float32, device="cuda")
    z = convnet.conv3x3(a.astype(np.float64), w, b.astype(np.float64))
    for act in (False, True):
        out = torch.empty((B, cout, H, W), dtype=torch.float32, device="cuda")
        es.es_nn_conv_forward(at, wt, torch.tensor(b, device="cuda"), out, act, ws)
        got, ref = out.cpu().double().numpy(), np.tanh(z) if act else z
        assert np.abs(got - ref).max() <= 4e-7 * np.sqrt(9 * cin) * np.abs(z).max()
        go = rng.standard_normal((B, cout, H, W)).astype(np.float32)
        g = torch.tensor(go, device="cuda")
        gin, gw, gb = torch.empty_like(at), torch.empty((cout, cin, 3, 3), device="cuda"), torch.empty(cout, device="cuda")
        es.es_nn_conv_backward(at, wt, out, g, gin, gw, gb, act, ws)
        gz = go * (1.0 - np.tanh(z) ** 2) if act else go.astype(np.float64)
        rw, rb, ra = convnet.conv3x3_backward(a.astype(np.float64), w, gz)
        # the layer's output enters the gradient through tanh with its own rounding: 4e-7 sqrt(n) of |z| in 1 - a^2
        back = 8e-7 * np.sqrt(9 * cin) * np.abs(z).max() if act else 0.0
        assert np.abs(g.cpu().double().numpy() - gz).max() <= (2e-7 + back) * np.abs(go).max()
        for got, ref, n in ((gw, rw, B * H * W), (gb, rb, B * H * W), (gin, ra, 9 * cout)):
            scale = np.abs(ref).max() + np.abs(go).max() * (np.abs(a).max() if ref is rw else 1.0)
            assert np.abs(got.cpu().double().numpy() - ref).max() <= (4e-7 * np.sqrt(n) + back * np.sqrt(n)) * scale


@pytest.mark.parametrize("cin", [2, 4, 32])
@pytest.mark.parametrize("cout", [2, 32])
def test_forward_infinite_and_nan_inputs(cin, cout):
    """An infinite input reaches the nine outputs whose taps read it as an infinity of the product's sign (tanh: +-1), a NaN
    as a NaN, and every other output as if they were zero."""
    import torch

    from paper_2407_05568_gb300 import es
    B, H, W = 2, 21, 35
    rng = np.random.default_rng(5 + cin + cout)
    a = rng.standard_normal((B, cin, H, W)).astype(np.float32)
    w = convnet.bf16_round((rng.standard_normal((cout, cin, 3, 3)) / np.sqrt(9 * cin)).astype(np.float32))
    assert (w != 0.0).all()
    zero = a.copy()
    spots = [(0, 0, 10, 14, np.inf), (0, cin - 1, 16, 24, -np.inf), (1, 1, 5, 5, np.nan), (1, 0, 15, 16, np.inf)]
    for b, c, y, x, v in spots:
        a[b, c, y, x], zero[b, c, y, x] = v, 0.0
    z = convnet.conv3x3(zero.astype(np.float64), w)
    size = np.abs(z).max()
    for b, c, y, x, v in spots:
        z[b, :, y - 1:y + 2, x - 1:x + 2] = (v * w[:, c, ::-1, ::-1]).reshape(cout, 3, 3)
    wt = torch.tensor(w, dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(es.es_nn_workspace_bytes(B, cin, cout, H, W) // 4 + 1, dtype=torch.float32, device="cuda")
    bias = torch.zeros(cout, device="cuda")
    for act in (False, True):
        out = torch.empty((B, cout, H, W), dtype=torch.float32, device="cuda")
        es.es_nn_conv_forward(torch.tensor(a, device="cuda"), wt, bias, out, act, ws)
        got, ref = out.cpu().double().numpy(), np.tanh(z) if act else z
        fin = np.isfinite(ref)
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
        assert np.abs(got[fin] - ref[fin]).max() <= 4e-7 * np.sqrt(9 * cin) * size


@pytest.mark.parametrize("cin", [2, 32])
@pytest.mark.parametrize("cout", [4, 32])
@pytest.mark.parametrize("where", ["input", "gradient"])
def test_weight_gradient_of_an_infinity(cin, cout, where):
    """One infinite value of the input, or of the output's gradient, away from the edges: the weight gradients that it
    enters are infinities of the product's sign, and the others stay finite and as accurate as without it."""
    import torch

    from paper_2407_05568_gb300 import es
    B, H, W, b, y, x, c = 1, 40, 37, 0, 18, 14, 1
    rng = np.random.default_rng(9 + cin + cout)
    a = rng.standard_normal((B, cin, H, W)).astype(np.float32)
    go = rng.standard_normal((B, cout, H, W)).astype(np.float32)
    w = convnet.bf16_round(rng.standard_normal((cout, cin, 3, 3)).astype(np.float32))
    a0, g0 = a.copy(), go.copy()
    (a0 if where == "input" else g0)[b, c, y, x] = 0.0
    (a if where == "input" else go)[b, c, y, x] = np.inf
    rw, rb, _ = convnet.conv3x3_backward(a0.astype(np.float64), w, g0.astype(np.float64))
    size = np.abs(rw).max()
    if where == "input":                                 # w[co][c][tap] takes g[co] at (y, x) less the tap
        rw[:, c] = np.inf * np.sign(go[b, :, y - 1:y + 2, x - 1:x + 2][:, ::-1, ::-1])
    else:
        rw[c] = np.inf * np.sign(a[b, :, y - 1:y + 2, x - 1:x + 2])
        rb[c] = np.inf
    at, g = torch.tensor(a, device="cuda"), torch.tensor(go, device="cuda")
    ws = torch.empty(es.es_nn_workspace_bytes(B, cin, cout, H, W) // 4 + 1, dtype=torch.float32, device="cuda")
    gw, gb = torch.empty((cout, cin, 3, 3), device="cuda"), torch.empty(cout, device="cuda")
    es.es_nn_conv_backward(at, torch.tensor(w, dtype=torch.bfloat16, device="cuda"), None, g, None, gw, gb, False, ws)
    for got, ref in ((gw.cpu().double().numpy(), rw), (gb.cpu().double().numpy(), rb)):
        fin = np.isfinite(ref)
        assert np.array_equal(got[~fin], ref[~fin])
        assert np.abs(got[fin] - ref[fin]).max() <= 4e-7 * np.sqrt(B * H * W) * (size + 1.0)


def test_forward_of_the_largest_floats():
    """Finite inputs that round to infinity in bf16 (above 3.39e38): the layer's output is their exact product."""
    import torch

    from paper_2407_05568_gb300 import es
    big = np.array([3.4028234e38, -3.4e38, 3.3961e38], np.float32)
    a = np.zeros((1, 4, 9, 9), np.float32)
    a[0, 2, 4, [1, 4, 7]] = big
    w = np.zeros((2, 4, 3, 3), np.float32)
    w[0, 2, 1, 1], w[1, 2, 1, 1] = 0.25, -0.5
    out = torch.empty((1, 2, 9, 9), dtype=torch.float32, device="cuda")
    ws = torch.empty(es.es_nn_workspace_bytes(1, 4, 2, 9, 9) // 4 + 1, dtype=torch.float32, device="cuda")
    es.es_nn_conv_forward(torch.tensor(a, device="cuda"), torch.tensor(w, dtype=torch.bfloat16, device="cuda"),
                          torch.zeros(2, device="cuda"), out, False, ws)
    got = out.cpu().numpy()[0, :, 4, [1, 4, 7]]
    ref = np.stack([0.25 * big, -0.5 * big], 1)
    assert np.all(np.abs(got.astype(np.float64) - ref) <= 2.0 ** -22 * np.abs(ref))


@pytest.mark.parametrize("shape", [(4, 512, 512), (3, 700, 530)])
def test_weight_gradient_of_long_strips(shape):
    """Strips of four 16-row tiles, whose two buffers are refilled several times (the training size, and a ragged image),
    against float64.  With R the root of the sum of squared products, about 150 rounded additions of partial sums of size R
    leave a random walk of 2^-24 sqrt(150) R = 7e-7 R; a dropped third part of one operand would leave 4e-6 R."""
    import torch

    from paper_2407_05568_gb300 import es
    B, H, W = shape
    gen = torch.Generator(device="cuda").manual_seed(H)
    a = torch.randn((B, 32, H, W), generator=gen, device="cuda")
    g = torch.randn((B, 32, H, W), generator=gen, device="cuda")
    w = torch.zeros((32, 32, 3, 3), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(es.es_nn_workspace_bytes(B, 32, 32, H, W) // 4 + 1, dtype=torch.float32, device="cuda")
    gw, gb = torch.empty((32, 32, 3, 3), device="cuda"), torch.empty(32, device="cuda")
    es.es_nn_conv_backward(a, w, None, g, None, gw, gb, False, ws)
    rw, r2 = torch.zeros((32, 32, 3, 3), dtype=torch.float64, device="cuda"), torch.zeros((32, 32, 3, 3), device="cuda")
    for b in range(B):
        ap, gd = torch.nn.functional.pad(a[b], (1, 1, 1, 1)), g[b].double().reshape(32, -1)
        for t in range(9):
            x = ap[:, t // 3:t // 3 + H, t % 3:t % 3 + W].reshape(32, -1)
            rw[:, :, t // 3, t % 3] += gd @ x.double().T
            r2[:, :, t // 3, t % 3] += (g[b].reshape(32, -1) ** 2) @ (x ** 2).T
    assert float(((gw.double() - rw).abs() / r2.sqrt()).max()) <= 2e-6
    rb = g.double().sum((0, 2, 3))
    assert float((gb.double() - rb).abs().max()) <= 2e-6 * (B * H * W) ** 0.5


def test_weight_gradient_of_a_tall_image():
    """A strip as tall as the image, 4096 rows: every product is (1 + d)(1 + e), whose leading parts are ones and sum
    exactly, so that the error is that of the correction products' sum.  Added to the rounded sum every 64 rows they leave
    the random walk of 64 half ulps, 2^-25 sqrt(64) = 2.4e-7, twice that at most."""
    import torch

    from paper_2407_05568_gb300 import es
    H, W = 4096, 16 * 1064                                       # as many strips as the grid takes: one per column
    x, g = np.float32(1.0037841), np.float32(1.0034173)
    a = torch.full((1, 2, H, W), float(x), device="cuda")
    go = torch.full((1, 2, H, W), float(g), device="cuda")
    ws = torch.empty(es.es_nn_workspace_bytes(1, 2, 2, H, W) // 4 + 1, dtype=torch.float32, device="cuda")
    gw, gb = torch.empty((2, 2, 3, 3), device="cuda"), torch.empty(2, device="cuda")
    es.es_nn_conv_backward(a, torch.zeros((2, 2, 3, 3), dtype=torch.bfloat16, device="cuda"), None, go, None, gw, gb, False, ws)
    assert abs(float(gw[1, 0, 1, 1]) / (float(x) * float(g) * H * W) - 1.0) <= 4.8e-7
    assert abs(float(gb[1]) / (float(g) * H * W) - 1.0) <= 4.8e-7


@pytest.mark.parametrize("cin,cout,shape", [(4, 32, (1, 16, 16)), (32, 32, (2, 50, 33)), (32, 2, (1, 64, 64))])
def test_backward_stays_in_its_workspace(cin, cout, shape):
    """The backward call with exactly the bytes that es_nn_workspace_bytes asks for: nothing behind them is written, and the
    gradients are those of a call with a larger workspace."""
    import torch

    from paper_2407_05568_gb300 import es
    B, H, W = shape
    gen = torch.Generator(device="cuda").manual_seed(cin + cout)
    a = torch.randn((B, cin, H, W), generator=gen, device="cuda")
    g = torch.randn((B, cout, H, W), generator=gen, device="cuda")
    w = torch.randn((cout, cin, 3, 3), generator=gen, device="cuda").to(torch.bfloat16)
    n = es.es_nn_workspace_bytes(B, cin, cout, H, W) // 4
    whole = torch.full((n + 4096,), 7.0, device="cuda")
    got = []
    for ws in (whole[:n], torch.empty(2 * n, device="cuda")):
        gw, gb, gin = torch.empty((cout, cin, 3, 3), device="cuda"), torch.empty(cout, device="cuda"), torch.empty_like(a)
        es.es_nn_conv_backward(a, w, None, g.clone(), gin, gw, gb, False, ws)
        got.append((gw, gb, gin))
    assert bool((whole[n:] == 7.0).all())
    assert all(torch.equal(p, q) for p, q in zip(*got))
