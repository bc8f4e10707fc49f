"""The autotuner's choice where the row layout over a cluster (schedule 64) is a
candidate: it shares the SMs among more rows, which a handle of a few rows does
not have, so those are tuned at their own number of rows."""
import math

import pytest

from helpers import to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402


def _masks(J, N):
    g = torch.Generator("cuda").manual_seed(N + J)
    return torch.polar(torch.ones(J, N, device="cuda"), 2 * math.pi * torch.rand(J, N, generator=g, device="cuda"))


@pytest.mark.parametrize("N,J", [(4096, 4), (4096, 6), (4096, 8), (2048, 6), (2048, 8)])
def test_few_rows_get_the_schedule_that_is_faster_for_them(N, J, tmp_path):
    d, cache = _masks(J, N), str(tmp_path / "tune.json")
    with tmr.tmr_create(N, 5000, J, d, None, dict(m=4, tune_cache=cache)) as h:  # the large matrix first
        many = tmr.tmr_schedule(h)
    with tmr.tmr_create(N, 8, J, d, None, dict(m=4, tune_cache=cache)) as h:
        few = tmr.tmr_schedule(h)
    assert many == 64 and few in (1, 2)  # measured 142 us against 206 for 8 rows, 1526 against 2579 for 608 (N = 4096, J = 4)
    for M, G in ((5000, many), (8, few)):  # both choices are kept, in memory and in the file
        with tmr.tmr_create(N, M, J, d, None, dict(m=4, tune_cache=cache)) as h:
            assert tmr.tmr_schedule(h) == G and tmr.tmr_autotune_report(h) == {}


def test_a_single_row_and_none():
    N, J = 4096, 4
    d = _masks(J, N)
    g = torch.Generator("cuda").manual_seed(3)
    T = torch.view_as_complex(torch.randn(1, N, 2, generator=g, device="cuda")) / math.sqrt(2 * N)
    Y = torch.fft.fft(d * T[:, None]).abs().square().contiguous()
    To, loss = torch.empty_like(T), torch.empty(1, device="cuda")
    with tmr.tmr_create(N, 1, J, d, None, {}) as h:
        assert tmr.tmr_schedule(h) == 1
        tmr.tmr_retrieve_from(h, T, Y, None, 1, To, None, None, loss)
        torch.cuda.synchronize()
    assert float((To - T).norm() / T.norm()) < 1e-4 and to_np(loss)[0] >= 0
    with tmr.tmr_create(N, 0, J, d, None, {}) as h:
        assert tmr.tmr_schedule(h) in (1, 64)
