"""Products of different shapes from several host threads at once: each runs the
same kernel with its own number of shared-memory stages, and none may be refused
or come out wrong because of another one's."""
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402


def test_threads_with_different_depths():
    # K = 64: two stages of the 32-column tile; K = 1024: ten
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    work, errors = [], []
    for K in (1024, 64, 64, 1024):
        A, B = (torch.randn(128, K, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
        work.append((A, B, torch.empty(128, 128, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    start = threading.Barrier(len(work))

    def run(A, B, C, stream):
        start.wait()
        try:
            for _ in range(2000):
                tmr.tmr_gemm_bf16(A, B, C, stream=stream.cuda_stream)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for A, B, C, _ in work:
        ref = A.double() @ B.double().T
        # FP32 sums of K products of unit variance
        assert float((C - ref).abs().max()) <= 1e-5 * A.shape[1]
