"""Networks whose layer widths are no multiples of 8 (the rows of the BF16
matrices are padded): values against a 64-bit network with the same roundings to
BF16, and the same kernels as their neighbours', seen by their time."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402

F64 = torch.float64


def _bf(x):
    return x.to(torch.bfloat16).to(F64)


def _layers(theta, dims):
    out, o = [], 0
    for a, b in zip(dims, dims[1:]):
        out.append((theta[o:o + a * b].reshape(b, a).to(F64), theta[o + a * b:o + a * b + b].to(F64)))
        o += a * b + b
    return out


def _reference(theta, dims, X, T):
    """Output and gradient in 64 bits with the library's roundings: operands of the products in BF16."""
    L, gelu = _layers(theta, dims), torch.nn.functional.gelu
    z, h = [], [_bf(X)]
    for i, (W, b) in enumerate(L):
        z.append(h[-1] @ _bf(W).T + b)
        if i < 2:
            h.append(_bf(gelu(z[-1])))
    d = _bf(2 * (z[-1] - T.to(F64)) / T.numel())
    grads = []
    for i in (2, 1, 0):
        grads.append(torch.cat([(d.T @ h[i]).flatten(), d.sum(0)]))
        if i:
            zi = z[i - 1]
            dgelu = 0.5 * (1 + torch.erf(zi / 2 ** 0.5)) + zi * torch.exp(-zi * zi / 2) / (2 * torch.pi) ** 0.5
            d = _bf((d @ _bf(L[i][0])) * dgelu)
    return z[-1], torch.cat(grads[::-1])


@pytest.mark.parametrize("dims,B", [((200, 132, 134, 130), 128), ((201, 129, 131, 133), 129), ((72, 260, 130, 402), 200),
                                    ((257, 128, 136, 131), 67), ((9, 7, 5, 3), 4)])
def test_values(dims, B):
    g = torch.Generator("cuda").manual_seed(sum(dims))
    X, T = (torch.randn(B, n, generator=g, device="cuda") for n in (dims[0], dims[3]))
    with tmr.tmr_mlp_create(*dims, seed=1) as net:
        theta = torch.randn(net.n_params, generator=g, device="cuda") * 0.1
        tmr.tmr_mlp_set_params(net, theta)
        Y, G, loss = torch.empty_like(T), torch.empty_like(theta), torch.empty(1, device="cuda")
        tmr.tmr_mlp_forward(net, X, B, Y)
        tmr.tmr_mlp_grad(net, X, T, B, loss, G)
        G2 = torch.empty_like(theta)
        tmr.tmr_mlp_train_step(net, X, T, B, 1e-3, loss)  # fused update: the next gradient sees the new weights
        after = torch.empty_like(theta)
        tmr.tmr_mlp_get_params(net, after)
        tmr.tmr_mlp_grad(net, X, T, B, loss, G2)
        torch.cuda.synchronize()
    # A value next to a rounding boundary may fall to its other side, one part
    # in 2^8 of that operand: of n terms a few do, which leaves the sum's relative
    # error well below 2^-8 / 4
    bar = 1e-3
    for th, grad in ((theta, G), (after, G2)):
        Yr, Gr = _reference(th, dims, X, T)
        if th is theta:
            assert float((Y - Yr).norm() / Yr.norm()) <= bar
        assert float((grad - Gr).norm() / Gr.norm()) <= bar
    # the first Adam step from zero moments: lr g / (|g| + 1e-8)
    step = 1e-3 * G.to(F64) / (G.to(F64).abs() + 1e-8)
    assert float((after - (theta.to(F64) - step)).abs().max()) <= 1e-6


def _step_us(dims, B):
    g = torch.Generator("cuda").manual_seed(0)
    X, T = (torch.randn(B, n, generator=g, device="cuda") for n in (dims[0], dims[3]))
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    with tmr.tmr_mlp_create(*dims, seed=1) as net:
        best = 1e9
        for _ in range(8):
            a.record()
            for _ in range(10):
                tmr.tmr_mlp_train_step(net, X, T, B, 1e-4)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 100)
    return best


@pytest.mark.parametrize("dims", [(8192, 132, 132, 4096), (9144, 1024, 1024, 4572), (4572, 1020, 1020, 2286)])
def test_odd_widths_run_on_the_same_kernels(dims):
    wide = tuple((n + 63) // 64 * 64 for n in dims)
    # on the generic kernel one of these steps takes 2 to 5 times as long as its neighbour
    assert _step_us(dims, 256) <= 1.6 * _step_us(wide, 256)
