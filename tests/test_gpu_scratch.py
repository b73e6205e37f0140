"""Device scratch of the compressed searches: the pool keeps what a search once took, so the key buffer has a cap."""
import pytest
import torch

from test_zz_no_alloc import _PoolWatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_counts", [False, True])
def test_keys_of_a_large_batch_stay_within_two_gigabytes(soar, own_counts):
    """Slices that do not fit side by side are packed; where they still do not fit, they take two passes."""
    g = torch.Generator(device="cuda").manual_seed(1)
    n, d, c, nq = 200_000, 16, 64, 1600
    X = torch.nn.functional.normalize(torch.randn(n, d, generator=g, device="cuda"), dim=1)
    Q = torch.nn.functional.normalize(torch.randn(nq, d, generator=g, device="cuda"), dim=1)
    tpq = torch.randint(-1, c + 2, (nq,), generator=g, device="cuda").int() if own_counts else None
    C = X[:c].contiguous()
    A = soar.soar_assign(X, C, 1.0, 1)
    ix = soar.soar_index_build(X, C, A, mode=soar.SOAR_SCORE_FP8)
    with _PoolWatch() as w:
        ids, sc = soar.soar_search(ix, Q, 10, c, tpq, rescore=200)   # every partition: 4 bytes x 2 n x nq = 2.56 GB
    # the other buffers: pairs, probe lists and centroid scores, well below 100 bytes a pair
    assert w.high - w.used0 <= 2 ** 31 + 100 * nq * c
    for q in range(0, nq, 400):
        part, part_sc = soar.soar_search(ix, Q[q:q + 400].contiguous(), 10, c,
                                         None if tpq is None else tpq[q:q + 400].contiguous(), rescore=200)
        assert torch.equal(ids[q:q + 400], part) and torch.equal(sc[q:q + 400], part_sc)
    ix.close()
