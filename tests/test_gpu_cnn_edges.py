"""The surrogate network beyond its accuracy at ordinary sizes: its state on creation, its memory, gradient
sums over many pixels and of extreme values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    import paper_2210_07501_gb300 as p
    p.build()
    p.load()
    return p


@pytest.mark.parametrize("own_stream", [False, True])
def test_new_network_runs_on_the_parameters_it_reports(pkg, own_stream):
    """A network reads its weights from copies laid out for the kernels; on creation, too, they are those
    of the parameters: outputs before any set_params are bit for bit those after putting the
    reported parameters back.  Many networks in a row, on a stream that nothing else orders."""
    x = torch.randn((1, 12, 17, 33), device="cuda")
    y0, y1 = (torch.empty((1, 4, 17, 33), device="cuda") for _ in range(2))
    for seed in range(20):
        stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
        torch.cuda.synchronize()
        net = pkg.Cnn(17, 33, batch_max=1, seed=seed, stream=stream)
        net.forward(x, y0)
        net.set_params(net.get_params())
        net.forward(x, y1)
        torch.cuda.synchronize()
        assert float(y0.abs().max()) > 0 and torch.equal(y0, y1), seed
        net.close()


@pytest.mark.parametrize("bf16,per_pixel", [(True, 752), (False, 1104)])
def test_device_memory_per_pixel(pkg, bf16, per_pixel):
    """What a network takes of the device grows by no more than 752 bytes a pixel with BF16 activations
    (every layer's output once, two gradients and 144 bytes of partial sums: images and batches that
    fit by that measure must keep fitting), 1104 with FP32's; and 64 MB whatever the size."""
    torch.cuda.synchronize()
    B, H, W = 8, 1024, 1024
    free = torch.cuda.mem_get_info()[0]
    net = pkg.Cnn(H, W, batch_max=B, bf16=bf16)
    used = free - torch.cuda.mem_get_info()[0]
    net.close()
    print(f"{used / (B * H * W):.0f} bytes a pixel")
    assert used <= per_pixel * B * H * W + (64 << 20)


CH = (12, 32, 32, 32, 32, 32, 4)


def exact_network(pkg, B, H, W, z=32.0):
    """A network (FP32 activations) whose gradients are known sums: the first layer's output is its
    bias z >= 32 (silu(z) = z and silu'(z) = 1 in FP32); the identity, then channel sums less 8 z: outputs
    zero.  With targets -d, every gradient is a sum of 2 d / (outputs) over pixels, times z in
    the weights behind the first layer (32 -> 32 layers: between equal channels too)."""
    net = pkg.Cnn(H, W, batch_max=B, bf16=False)
    p = []
    for l in range(6):
        ci, co = CH[l], CH[l + 1]
        w, b = np.zeros((co, ci, 3, 3), np.float32), np.zeros(co, np.float32)
        if l == 0:
            b[:] = z
        elif l < 5:
            w[np.arange(co), np.arange(ci), 1, 1] = 1.0
        else:
            w[np.arange(ci) % co, np.arange(ci), 1, 1] = 1.0
            b[:] = -8.0 * z
        p += [w.ravel(), b]
    net.set_params(np.concatenate(p))
    return net


def layers_of(grad):
    out, o = [], 0
    for l in range(6):
        n = CH[l] * CH[l + 1] * 9
        out.append((grad[o:o + n].reshape(CH[l + 1], CH[l], 3, 3), grad[o + n:o + n + CH[l + 1]]))
        o += n + CH[l + 1]
    return out


def test_weight_gradients_over_many_tiles(pkg):
    """4.2 M pixels, 16384 tiles of the weight gradient, ~54 a CTA.  dz is one number whose sums over a tile are
    exact in FP32, so what is measured is the sum over the tiles: as good as FP64's, rounded once per
    CTA and once at the end (2^-24 each).  Summed in FP32 over a CTA's tiles it is 4e-7 off."""
    B, H, W = 16, 512, 512
    net = exact_network(pkg, B, H, W)
    d = 5020203 / 2.0 ** 23
    x = torch.ones((B, 12, H, W), device="cuda")
    t = torch.full((B, 4, H, W), -d, device="cuda")
    grad, _ = net.gradients(x, t)
    net.close()
    dz = 2.0 * d / (B * 4 * H * W)
    full, edge = dz * B * H * W, dz * B * (H - 1) * W     # a tap in the row, in the row above or below
    taps = np.array([edge, full, edge])[:, None] * np.ones((1, 3))
    worst = 0.0
    for l, (w, b) in enumerate(layers_of(grad.astype(np.float64))):
        expect = taps * (1.0 if l == 0 else 32.0)
        worst = max(worst, np.max(np.abs(w / expect - 1.0)), np.max(np.abs(b / full - 1.0)))
    print(f"largest relative error of a gradient: {worst:.2e}")
    assert worst <= 1.3e-7


def test_weight_gradients_of_extreme_values(pkg):
    """An infinite dz makes the gradients it enters infinite and no others NaN; sums that overflow FP32 on the
    way and not in the end (128 tiles, half of them +, half -) come out as in FP64: zero."""
    H, W = 8, 32 * 128
    net = exact_network(pkg, 1, H, W, z=128.0)
    x = torch.ones((1, 12, H, W), device="cuda")
    t = torch.zeros((1, 4, H, W), device="cuda")
    t[0, 1, 3, 700] = -float("inf")
    w, b = layers_of(net.gradients(x, t)[0])[5]
    for a in (w, b):
        assert np.all(np.isposinf(a[1])) and np.all(a[[0, 2, 3]] == 0.0)
    t[:, :, :, : W // 2], t[:, :, :, W // 2:] = -1.7e38, 1.7e38
    w, b = layers_of(net.gradients(x, t)[0])[5]
    net.close()
    assert np.all(w == 0.0) and np.all(b == 0.0)
