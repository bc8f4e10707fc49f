"""The row layout over a cluster of CTAs asked for by its code (opt.schedule =
64), so that no test hangs on what the autotuner picks: more iterations than the
L-BFGS memory holds (the oldest pair is dropped), rows that stop early, and
starts proposed by a network, each against one mask per CTA (schedule 1) on the
same rows, the drop against the FP64 oracle too."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_rows_close, c64, f32, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402

SHAPES = [(4096, 4), (4096, 6), (4096, 8), (2048, 6), (2048, 8)]


def _problem(N, M, J, seed):
    T = c64(synth.tm_iid(M, N, seed=seed))
    d = c64(synth.mask_phases(J, N, seed=seed)[1])
    y = torch.empty((M, J, N), dtype=torch.float32, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d), None, dict(schedule=1)) as h:
        tmr.tmr_forward(h, to_dev(T), y)
    return T, d, y


def _run(G, N, M, J, d, y, iters, T_init=None, model=None, **opt):
    To = torch.empty((M, N), dtype=torch.complex64, device="cuda")
    st, it = (torch.empty(M, dtype=torch.int32, device="cuda") for _ in range(2))
    with tmr.tmr_create(N, M, J, to_dev(d), None, dict(opt, schedule=G)) as h:
        assert tmr.tmr_schedule(h) == G
        if model is not None:
            tmr.tmr_set_init_model(h, model)
        if T_init is None:
            tmr.tmr_retrieve(h, y, None, iters, To, st, it)
        else:
            tmr.tmr_retrieve_from(h, to_dev(T_init), y, None, iters, To, st, it)
        torch.cuda.synchronize()
        kept = tmr.tmr_learned_rows(h) if model is not None else 0
    return to_np(To), to_np(st), to_np(it), kept


@pytest.mark.parametrize("N,J", SHAPES)
def test_every_reported_code_can_be_given_back(N, J):
    d = to_dev(c64(synth.mask_phases(J, N, seed=0)[1]))
    with tmr.tmr_create(N, 200, J, d, None, {}) as h:
        code = tmr.tmr_schedule(h)
    with tmr.tmr_create(N, 200, J, d, None, dict(schedule=code)) as h:
        assert tmr.tmr_schedule(h) == code


def test_shapes_without_the_layout_are_refused():
    for N, J, opt in ((1024, 4, {}), (2048, 4, {}), (2048, 5, {}), (4096, 2, {}), (4096, 4, dict(cost="amplitude")),
                      (4096, 4, dict(m=6)), (4096, 4, dict(precision="mixed"))):
        d = to_dev(np.ones((J, N), np.complex64))
        with pytest.raises(tmr.TMRError) as ei:
            tmr.tmr_create(N, 4, J, d, None, dict(opt, schedule=64))
        assert ei.value.status == tmr.TMR_ERR_UNSUPPORTED


@pytest.mark.parametrize("N,J,m", [(N, J, 2) for N, J in SHAPES] + [(4096, 4, 5), (2048, 6, 6)])
def test_dropping_the_oldest_pair(N, J, m):
    M, iters = 90, m + 3  # more rows than clusters
    T, d, y = _problem(N, M, J, seed=N + J + m)
    T0 = c64(T + 0.1 * synth.tm_iid(M, N, seed=1))
    A, sa, ia, _ = _run(64, N, M, J, d, y, iters, T0, m=m)
    B, sb, ib, _ = _run(1, N, M, J, d, y, iters, T0, m=m)
    assert np.array_equal(sa, sb) and np.array_equal(ia, ib) and np.all(ia == iters)
    # two FP32 solvers, each within 1e-4 a step of the oracle
    assert_rows_close(A, B.astype(np.complex128), 2e-4 * iters)


@pytest.mark.parametrize("N,J", [(4096, 4), (2048, 6)])
def test_dropping_matches_the_oracle(N, J):
    M, m, iters = 2, 2, 5
    T, d, y = _problem(N, M, J, seed=11)
    T0 = c64(T + 0.1 * synth.tm_iid(M, N, seed=2))
    A, _, _, _ = _run(64, N, M, J, d, y, iters, T0, m=m)
    Tr, _, _, _ = oracle.retrieve_rows(to_np(y), d.astype(np.complex128), iters, m=m, T_init=T0)
    assert_rows_close(A, Tr, 1e-4 * iters)


@pytest.mark.parametrize("N,J", [(4096, 4), (2048, 8)])
def test_rows_that_stop_early(N, J):
    M, iters = 90, 60
    T, d, y = _problem(N, M, J, seed=5)
    step = 10.0 ** np.random.default_rng(0).uniform(-3, -0.7, size=(M, 1))  # rows at other distances
    T0 = c64(T + step * synth.tm_iid(M, N, seed=3))
    y = y * (1 + 0.01 * torch.randn(y.shape, generator=torch.Generator("cuda").manual_seed(0), device="cuda"))
    A, sa, ia, _ = _run(64, N, M, J, d, y, iters, T0, tol=1e-3)
    B, sb, ib, _ = _run(1, N, M, J, d, y, iters, T0, tol=1e-3)
    assert np.all(sa == 1) and np.all(sb == 1) and ia.min() < ia.max() < iters
    # a row whose last decrease stands at the bar may take one step more on one side
    assert np.max(np.abs(ia - ib)) <= 1 and np.mean(ia == ib) > 0.9
    same = ia == ib
    assert_rows_close(A[same], B[same].astype(np.complex128), 2e-4 * iters)


@pytest.mark.parametrize("power_iters", [0, 6])
def test_starts_from_a_network(power_iters):
    N, J, M, iters = 2048, 6, 90, 2
    T, d, y = _problem(N, M, J, seed=9)
    opt = dict(init="learned", power_iters=power_iters)
    with tmr.tmr_mlp_create(J * N, 64, 64, 2 * N, seed=5) as net:
        A, sa, ia, ka = _run(64, N, M, J, d, y, iters, model=net, **opt)
        B, sb, ib, kb = _run(1, N, M, J, d, y, iters, model=net, **opt)
    assert np.array_equal(sa, sb) and np.array_equal(ia, ib) and ka == kb
    # six products and two steps on rows far from convergence amplify FP32's 1e-6 by less than 100
    assert_rows_close(A, B.astype(np.complex128), 1e-4)
