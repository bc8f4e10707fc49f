"""The one-CTA-per-row solver with its fields in tensor memory, at the edges of
the rule that puts them there: pairs and fields fill all 512 columns (N = 2048
with J = 4, m = 5 and J = 2, m = 6), the first shapes that keep them in registers
(m = 6 at J = 4, m = 5 at J = 3), one to eight masks, both costs; against one mask
per CTA (schedule 1), the same iteration with other summation orders."""
import numpy as np
import pytest

import synth
from helpers import c64, assert_rows_close, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402


def _run(N, M, J, d, y, T_init, iters, **opt):
    To = torch.empty((M, N), dtype=torch.complex64, device="cuda")
    st, it = (torch.empty(M, dtype=torch.int32, device="cuda") for _ in range(2))
    loss = torch.empty(M, dtype=torch.float32, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d), None, opt) as h:
        tmr.tmr_retrieve_from(h, T_init, y, None, iters, To, st, it, loss)
        torch.cuda.synchronize()
    return to_np(To), to_np(st), to_np(it), to_np(loss)


# eight steps: more than the pairs of any m, so that the oldest is dropped
@pytest.mark.parametrize("N,J,m", [(2048, 4, 5), (2048, 4, 6), (2048, 3, 5), (2048, 3, 4), (2048, 2, 6),
                                   (1024, 8, 6), (1024, 4, 5), (1024, 4, 6), (1024, 5, 1), (512, 8, 5), (512, 4, 6),
                                   (512, 1, 6)])
@pytest.mark.parametrize("cost", ["intensity", "amplitude"])
def test_fields_in_tensor_memory(N, J, m, cost):
    M, iters = 200, 8  # more rows than CTAs of the largest shapes
    T = c64(synth.tm_iid(M, N, seed=N + J))
    d = c64(synth.mask_phases(J, N, seed=m)[1])
    y = torch.empty((M, J, N), dtype=torch.float32, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d), None, dict(schedule=1)) as h:
        tmr.tmr_forward(h, to_dev(T), y)
    y[3] = 0.0  # a dark row
    T_init = to_dev(c64(T + 0.2 * synth.tm_iid(M, N, seed=1)))
    A, sa, ia, la = _run(N, M, J, d, y, T_init, iters, m=m, cost=cost, schedule=16)
    B, sb, ib, lb = _run(N, M, J, d, y, T_init, iters, m=m, cost=cost, schedule=1)
    assert np.array_equal(sa, sb) and np.array_equal(ia, ib)
    assert not A[3].any()
    keep = np.arange(M) != 3
    # 1e-4 a step, as the steps of the other layouts are held to
    assert_rows_close(A[keep], B[keep].astype(np.complex128), 1e-4 * iters)
