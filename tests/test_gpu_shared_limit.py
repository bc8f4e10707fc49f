"""Problems whose row state fills the shared memory of an SM to the last few
bytes: they are taken, and solved, as any other (one step against the FP64
oracle).  The shapes come from the sizes of the row state alone; a state 28
bytes larger would refuse the first group, 32 bytes of static shared memory
beside it would fail the second at its launch."""
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

AT_THE_LIMIT = [(1564, 1, 4, 1), (2469, 2, 2, 32), (2963, 2, 1, 1), (4003, 6, 3, 1), (4088, 5, 2, 1)]
JUST_BELOW = [(2333, 3, 5, 1), (2587, 4, 6, 1), (3695, 3, 1, 1), (4087, 5, 2, 1)]


@pytest.mark.parametrize("N,J,m,G", AT_THE_LIMIT + JUST_BELOW)
def test_a_full_shared_memory_is_enough(N, J, m, G):
    M, iters = 2, 1
    T = c64(synth.tm_iid(M, N, seed=N))
    d = c64(synth.mask_phases(J, N, seed=N)[1])
    Y = f32(oracle.forward(T.astype(np.complex128), d.astype(np.complex128)))
    T0 = c64(T + 0.2 * synth.tm_iid(M, N, seed=1))
    To = torch.empty((M, N), dtype=torch.complex64, device="cuda")
    with tmr.tmr_create(N, M, J, to_dev(d), None, dict(schedule=G, m=m)) as h:
        assert tmr.tmr_schedule(h) == G
        tmr.tmr_retrieve_from(h, to_dev(T0), to_dev(Y), None, iters, To)
        torch.cuda.synchronize()
    Tr, _, _, _ = oracle.retrieve_rows(Y, d.astype(np.complex128), iters, T_init=T0, m=m)
    assert_rows_close(to_np(To), Tr, 1e-4)
