"""The row layout over a cluster of CTAs (schedule 64: N = 4096 with J = 4, 6, 8
and N = 2048 with J = 6, 8; slices of the vectors of unequal length at J = 6,
N = 4096) against one mask per CTA (schedule 1): the same iteration with other
summation orders, so the starts and a few steps agree to FP32 rounding, and
against the FP64 oracle.  The autotuner chooses the schedule; a row of the
matrix is skipped here if it chose another one."""
import numpy as np
import pytest

import oracle
import synth
from helpers import c64, f32, assert_rows_close, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402

SHAPES = [(4096, 4), (4096, 6), (4096, 8), (2048, 6), (2048, 8)]


def _problem(N, M, J, seed):
    T = c64(synth.tm_iid(M, N, seed=seed))
    d = c64(synth.mask_phases(J, N, seed=seed)[1])
    return T, d


def _run(N, M, J, d, y, iters, T_init=None, **opt):
    To = torch.empty((M, N), dtype=torch.complex64, device="cuda")
    st, it = (torch.empty(M, dtype=torch.int32, device="cuda") for _ in range(2))
    loss = torch.empty(M, dtype=torch.float32, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d), None, opt) as h:
        sched = tmr.tmr_schedule(h)
        if T_init is None:
            tmr.tmr_retrieve(h, y, None, iters, To, st, it, loss)
        else:
            tmr.tmr_retrieve_from(h, T_init, y, None, iters, To, st, it, loss)
        torch.cuda.synchronize()
    return sched, to_np(To), to_np(st), to_np(it), to_np(loss)


@pytest.mark.parametrize("N,J", SHAPES)
@pytest.mark.parametrize("start", ["given", "bp", "random", "power", "lanczos"])
def test_matches_one_mask_per_cta(N, J, start):
    M, iters = 90, 3  # more rows than clusters
    T, d = _problem(N, M, J, seed=N + J)
    y = torch.empty((M, J, N), dtype=torch.float32, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d), None, dict(schedule=1)) as h:
        tmr.tmr_forward(h, to_dev(T), y)
    y[3] = 0.0  # a dark row
    opt = dict(init={"power": "spectral", "lanczos": "spectral", "given": "random"}.get(start, start),
               power_iters=10, lanczos=int(start == "lanczos"))
    T_init = to_dev(c64(T + 0.2 * synth.tm_iid(M, N, seed=1))) if start == "given" else None
    sched, A, sa, ia, la = _run(N, M, J, d, y, iters, T_init, **opt)
    if sched != 64:
        pytest.skip(f"the autotuner chose schedule {sched}")
    _, B, sb, ib, lb = _run(N, M, J, d, y, iters, T_init, schedule=1, **opt)
    assert np.array_equal(sa, sb) and np.array_equal(ia, ib)
    assert not A[3].any()
    keep = np.arange(M) != 3
    # FP32 transforms agree to 1e-6; the start's ten products and three steps
    # on rows far from convergence amplify that by less than 100
    assert_rows_close(A[keep], B[keep].astype(np.complex128), 1e-4)
    assert np.max(np.abs(la[keep] - lb[keep]) / lb[keep]) <= 1e-3


@pytest.mark.parametrize("N,J", [(4096, 4), (2048, 6)])
def test_steps_match_the_oracle(N, J):
    M, iters = 2, 3
    T, d = _problem(N, M, J, seed=7)
    Y = f32(oracle.forward(T.astype(np.complex128), d.astype(np.complex128)))
    T_init = c64(T + 0.2 * synth.tm_iid(M, N, seed=2))
    sched, A, _, _, _ = _run(N, M, J, d, to_dev(Y), iters, to_dev(T_init))
    if sched != 64:
        pytest.skip(f"the autotuner chose schedule {sched}")
    Tr, _, _, _ = oracle.retrieve_rows(Y, d.astype(np.complex128), iters, T_init=T_init)
    assert_rows_close(A, Tr, 1e-4 * iters)
