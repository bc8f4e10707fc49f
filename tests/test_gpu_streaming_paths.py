"""The forward model, gradient and network paths that a call's sizes select,
at the edges of each, against the FP64 oracle: 16 points per thread for many
rows of a power of two, the composite lengths N = A B, the GEMM's epilogues and
K-strided operands, and the preprocessing's threshold search beyond the keys
that fit in shared memory."""
import numpy as np
import pytest

import oracle
import synth
from helpers import c64, assert_rows_close, to_dev, to_np
from oracle import mlp as omlp
from oracle import preprocess as pp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402


def _forward_and_grad(N, M, J, rows):
    """Library results of all M rows, the oracle's of `rows`, at the bound of
    the FP32 transforms (1e-5) that every length is held to."""
    T = c64(synth.tm_iid(M, N, seed=N))
    d = c64(synth.mask_phases(J, N, seed=M)[1])
    dd, Td = d.astype(np.complex128), T[rows].astype(np.complex128)
    Y = torch.empty((M, J, N), dtype=torch.float32, device="cuda")
    loss = torch.empty(M, dtype=torch.float32, device="cuda")
    G = torch.empty((M, N), dtype=torch.complex64, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d)) as h:
        tmr.tmr_forward(h, to_dev(T), Y)
        Yo = Y.roll(1, 0).contiguous()  # another row's intensities: large residuals
        tmr.tmr_grad(h, to_dev(T), Yo, loss, G)
        torch.cuda.synchronize()
    assert_rows_close(to_np(Y)[rows], oracle.forward(Td, dd), 1e-5)
    lo, Go = oracle.loss_grad(Td, dd, to_np(Yo)[rows].astype(np.float64))
    assert np.max(np.abs(to_np(loss)[rows] - lo) / lo) <= 1e-5
    assert_rows_close(to_np(G)[rows], Go, 1e-5)


# 608 transforms side by side are the line between 8 and 16 points per thread
@pytest.mark.parametrize("N,M,J", [(512, 151, 4), (512, 152, 4), (1024, 607, 1), (1024, 608, 1), (2048, 609, 3),
                                   (4096, 613, 2)])
def test_many_rows_of_a_power_of_two(N, M, J):
    _forward_and_grad(N, M, J, np.array([0, M // 2, M - 1]))


# A = 1 .. 32 (each team count and its neighbours), B up to 128; 131 and 4095 have no such split
@pytest.mark.parametrize("N", [18, 96, 129, 130, 131, 254, 381, 512 + 128, 9 * 113, 12 * 127, 13 * 128, 17 * 127,
                               18 * 128, 19 * 109, 24 * 125, 25 * 128, 31 * 128, 32 * 127, 4095])
def test_composite_lengths(N):
    _forward_and_grad(N, 5, 3, np.arange(5))


# rows of the composite lengths beyond one wave of CTAs
def test_composite_length_many_rows():
    _forward_and_grad(254, 9001, 2, np.array([0, 4500, 9000]))


def _adam_reference(theta, g, lr):
    z = np.zeros_like(theta)
    return omlp.adam_step(theta, g, z, z, 1, lr=lr)[0]


# B odd (a K tail of the weight gradients), 130 outputs (rows of the product not
# a multiple of four), widths off the tile, and every product on the tensor cores
@pytest.mark.parametrize("dims,B", [((256, 136, 128, 320), 133), ((128, 128, 128, 130), 160), ((264, 200, 136, 128), 300)])
@pytest.mark.parametrize("loss_kind", ["mse", "phase"])
def test_network_on_the_tensor_cores(dims, B, loss_kind):
    """Gradient against the oracle at the BF16 bound (8-bit mantissa operands,
    as test_gpu_learned); the training step's weights against the oracle's
    Adam on the library's own gradient at FP32 rounding of the update."""
    rng = np.random.default_rng(sum(dims) + B)
    lr = 3e-3
    with tmr.tmr_mlp_create(*dims, seed=3) as m:
        tmr.tmr_mlp_set_loss(m, loss_kind)
        theta = (rng.standard_normal(m.n_params) * 0.1).astype(np.float32)
        tmr.tmr_mlp_set_params(m, theta)
        X = rng.standard_normal((B, dims[0])).astype(np.float32)
        T = rng.standard_normal((B, dims[3])).astype(np.float32)
        G = torch.empty(m.n_params, dtype=torch.float32, device="cuda")
        loss = torch.empty(1, dtype=torch.float32, device="cuda")
        tmr.tmr_mlp_grad(m, to_dev(X), to_dev(T), B, loss, G)
        new = np.empty(m.n_params, np.float32)
        tmr.tmr_mlp_train_step(m, to_dev(X), to_dev(T), B, lr, loss)
        tmr.tmr_mlp_get_params(m, new)
        torch.cuda.synchronize()
    g = to_np(G)
    if loss_kind == "mse":
        Lo, Go = omlp.loss_grad(theta.astype(np.float64), dims, X, T)
        assert abs(float(to_np(loss)[0]) - Lo) <= 2e-2 * Lo
        assert np.linalg.norm(g - Go) <= 3e-2 * np.linalg.norm(Go)
    ref = _adam_reference(theta.astype(np.float64), g.astype(np.float64), lr)
    assert np.all(np.abs(new - ref) <= 1e-6 * np.abs(ref) + 1e-4 * lr)


# more pixels than keys fit in shared memory: 213,000 over the cluster, 26,000 in one CTA
@pytest.mark.parametrize("K,H,W,dtype", [(3, 1000, 900, np.uint16), (5, 330, 330, np.float32), (70, 129, 255, np.uint16)])
def test_threshold_search_of_large_grids(K, H, W, dtype):
    fr = synth.camera_frames(K, H, W, seed=K, dtype=dtype)
    out = tmr.preprocess(to_dev(fr.view(np.int16)) if dtype == np.uint16 else to_dev(fr))
    torch.cuda.synchronize()
    y, mask, E = pp.camera_rows(fr, 0, 0.999)
    assert np.array_equal(to_np(out["mask"]).astype(bool), mask) and int(out["n_inside"].item()) == int(mask.sum())
    np.testing.assert_allclose(to_np(out["energy"]), E, rtol=1e-13, atol=0)
    assert np.array_equal(to_np(out["y"]), y)


# equal energies: no bit of the FP64 keys differs
def test_threshold_search_of_equal_pixels():
    out = tmr.preprocess(torch.full((4, 10, 10), 3.0, device="cuda"))
    assert int(out["n_inside"].item()) == 25 and bool(out["mask"].all())
