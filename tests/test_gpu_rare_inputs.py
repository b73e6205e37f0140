"""Inputs off the beaten track: rows that are not numbers, clusters tighter than the screening bands, rows of very
uneven length."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d", [24, 160, 400])        # both tensor-core shapes and the general kernels
@pytest.mark.parametrize("spills", [0, 1, 2])
def test_points_without_a_number_are_assigned_nowhere(soar, dtype, d, spills):
    g = torch.Generator().manual_seed(d)
    X = torch.randn(300, d, generator=g).to(dtype)
    C = torch.randn(70, d, generator=g)
    want = soar.soar_assign(X.cuda(), C.cuda(), 1.0, spills)
    bad = torch.tensor([0, 17, 128, 299])
    X[bad, d // 2] = float("nan")
    got = soar.soar_assign(X.cuda(), C.cuda(), 1.0, spills)
    rest = torch.ones(300, dtype=torch.bool)
    rest[bad] = False
    assert torch.equal(got[rest.cuda()], want[rest.cuda()])
    assert (got[bad.cuda()] == -1).all()
