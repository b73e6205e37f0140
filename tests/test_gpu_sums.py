"""The k-means update's sums against exact ones, on members that cancel."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("decades", [7, 9, 12])
def test_centroid_sums_of_cancelling_members(soar, decades):
    """Each of the four interleaved partial sums of a 64-row cluster takes sixteen rows whose values span `decades`
    and nearly cancel, so that what remains is below the rounding errors of a plain fp32 sum.  The update carries
    those errors: it may lose 2^-59 of the summed magnitudes per partial sum (one batch of sixteen rows), and 2^-24
    of the result to its rounding."""
    d = 256
    g = torch.Generator().manual_seed(decades)
    V = torch.randn(4, 16, d, generator=g) * 10.0 ** (-decades * torch.rand(4, 16, d, generator=g))
    for last in (14, 15):
        for chain in range(4):
            for col in range(d):
                V[chain, last, col] = -math.fsum(V[chain, :last, col].tolist())
    X = V.transpose(0, 1).reshape(64, d).contiguous()            # row i belongs to partial sum i % 4
    C = soar.soar_train_centroids(X.cuda(), 1, 1, torch.zeros(1, dtype=torch.int32).cuda()).cpu()[0]
    for col in range(d):
        v = X[:, col].tolist()
        want, mag = math.fsum(v) / 64, sum(abs(x) for x in v) / 64
        assert abs(C[col].item() - want) <= 2.0 ** -57 * mag + 2.0 ** -23 * abs(want)
