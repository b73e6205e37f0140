"""Host threads that call one kernel with different shared-memory sizes."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(calls, rounds):
    """Each call `rounds` times in a thread and on a stream of its own; the exceptions raised."""
    errors = []

    def work(call):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(rounds):
                    call()
                torch.cuda.current_stream().synchronize()
        except Exception as e:                       # noqa: BLE001 (reported by the caller)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def test_searches_of_different_sizes_from_two_threads(soar):
    g = torch.Generator(device="cuda").manual_seed(1)
    n, d, c = 20_000, 32, 50
    X = torch.randn(n, d, generator=g, device="cuda")
    Q = torch.randn(64, d, generator=g, device="cuda")
    C = X[:c].contiguous()
    A = soar.soar_assign(X, C, 1.0, 1)
    fp8 = soar.soar_index_build(X, C, A, mode=soar.SOAR_SCORE_FP8)
    full = soar.soar_index_build(X, C, A)
    assert not _run([lambda: soar.soar_search(fp8, Q, 10, 8, rescore=10),
                     lambda: soar.soar_search(fp8, Q, 40, 8, rescore=4096)], 400)
    assert not _run([lambda: soar.soar_search(full, Q, 17, 8), lambda: soar.soar_search(full, Q, 128, 8)], 200)
    assert not _run([lambda: soar.soar_search(full, Q, 129, 8), lambda: soar.soar_search(full, Q, 700, 8)], 60)
    fp8.close()
    full.close()
