"""The persistent tensor-core convolution over its tile schedule, against the
same products in 64 bits on operands rounded to BF16.

What the kernel can get wrong at a schedule's edges is a whole tile or a whole
channel block, so it is held to the FP32 accumulation's own bound: K products of
BF16 values, exact in FP32, summed by the tensor cores with at most one
truncation (2^-22 of the running sum's magnitude) per product, and one rounding
for the bias: (K 2^-22) sum |a b| + 2^-23 |y|. Shapes: more tiles than SMs and
one more than a whole wave, weights resident and streamed through the ring
(beyond 128 outputs, and 256 x 128 channels), single rows and odd rows, widths
around one 128-pixel tile. The fused relu is compared bit for bit."""
import pytest

from gpu_common import package, torch_cuda

pytestmark = pytest.mark.gpu

SHAPES = [(1, 20, 32, 307, 100), (2, 33, 64, 153, 129), (1, 128, 64, 8, 127), (1, 256, 128, 5, 257),
          (1, 40, 300, 7, 128), (3, 1, 1, 103, 1)]


@pytest.mark.parametrize("shape", SHAPES)
def test_conv_tc_over_the_tile_schedule(shape):
    P = package()
    torch = torch_cuda()
    B, Ci, Co, H, W = shape
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    r = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16).to(torch.float32)  # noqa: E731
    x, w, b = r(B, Ci, H, W), r(Co, Ci, 3, 3), r(Co)
    y = torch.full((B, Co, H, W), float("nan"), device="cuda")
    z = torch.full_like(y, float("nan"))
    P.dg_nn_conv3x3_forward_tc(x, w, b, y)
    P.dg_nn_conv3x3_forward_tc(x, w, b, z, relu=True)
    h = torch.empty_like(y)
    P.dg_nn_relu_forward(y, h)
    P.dg_nn_tc_check()

    def conv(a, k):  # 64 bits, one shifted product per tap
        p = torch.nn.functional.pad(a.double(), (1, 1, 1, 1))
        out = torch.zeros((B, Co, H, W), dtype=torch.float64, device="cuda")
        for u in range(3):
            for v in range(3):
                out += torch.einsum("nchw,oc->nohw", p[:, :, u:u + H, v:v + W], k[:, :, u, v].double())
        return out

    ref = conv(x, w) + b.double().view(1, -1, 1, 1)
    lim = 9 * Ci * 2.0 ** -22 * conv(x.abs(), w.abs()) + 2.0 ** -23 * ref.abs() + 1e-30
    assert bool(((y.double() - ref).abs() <= lim).all())
    assert torch.equal(z, h)


@pytest.mark.parametrize("channels,shape", [([3, 1], (2, 9, 40)), ([20, 32, 1], (1, 33, 130)),
                                            ([5, 40, 130, 24, 1], (2, 7, 129)),
                                            ([7, 32, 64, 160, 32, 1], (3, 21, 257)), ([4, 96, 32, 1], (2, 1, 1)),
                                            ([33, 128, 64, 1], (1, 130, 128))])
def test_network_in_one_call_is_its_layers_one_by_one(channels, shape):
    from paper_2508_06672_gb300.proposal import ProposalNet
    P = package()
    torch = torch_cuda()
    net = ProposalNet(channels, seed=4, tc=True)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(shape[0], channels[0], *shape[1:], generator=g, device="cuda")
    h = x
    for k, (w, b) in enumerate(net.params):
        z = torch.empty((shape[0], channels[k + 1], *shape[1:]), device="cuda")
        P.dg_nn_conv3x3_forward_tc(h, w, b, z, relu=k + 1 < len(net.params))
        h = z
    y = net.forward(x)
    P.dg_nn_tc_check()
    assert torch.equal(y, h)
    assert torch.equal(net.forward(x, keep=True), h)


def _network():
    from paper_2508_06672_gb300.proposal import ProposalNet
    torch = torch_cuda()
    net = ProposalNet([20, 32, 64, 32, 1], seed=5, tc=True)
    x = torch.randn(1, 20, 129, 150, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    return torch, package(), net, x


def test_network_on_a_stream_of_its_own():
    """The call on another stream than the current one: its scratch and output belong
    to that stream, so nothing allocated meanwhile takes their place before the
    kernels, held up behind other work, have run."""
    torch, P, net, x = _network()
    ref = P.dg_nn_forward_tc(x, net.params)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(50_000_000)
    y = P.dg_nn_forward_tc(x, net.params, stream=s)
    held = [torch.full((n,), float("nan"), device="cuda") for n in (1 << 14, 1 << 17, 1 << 20, 1 << 21, 1 << 22) for _ in range(3)]
    torch.cuda.current_stream().synchronize()
    s.synchronize()
    assert torch.equal(y, ref)
    del held


def test_network_under_capture():
    """The network's launches, each let in before the one before it ends, recorded
    in a graph: replays give the call's output, also on new inputs."""
    torch, P, net, x = _network()
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        for _ in range(2):
            net.forward(x)
    torch.cuda.current_stream().wait_stream(s)
    with torch.cuda.graph(g):
        y = net.forward(x)
    for seed in (6, 7, 8):
        x.copy_(torch.randn(x.shape, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda"))
        y.zero_()
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, net.forward(x))
    P.dg_nn_tc_check()
