"""Edges of the rules that choose a kernel or its shape, against fp64 references."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,d,c", [
    (19_456, 64, 300), (19_457, 64, 300),           # one and two operands on 152 SMs
    (20_000, 5, 130), (20_000, 104, 257), (20_000, 152, 300),     # several items a block; 16-byte and single loads
    (16_384, 304, 64), (16_385, 304, 64), (3000, 304, 65),        # wide rows: general kernels up to 16 384 x 64
    (16_384, 150, 64), (3000, 150, 65),
])
def test_assignment_rules(soar, dtype, n, d, c):
    g = torch.Generator().manual_seed(n + d)
    X = torch.randn(n, d, generator=g).to(dtype).cuda()
    C = torch.randn(c, d, generator=g).cuda()
    A = soar.soar_assign(X, C, 1.5, 1).long()
    x, cc = X.double(), C.double()
    dist = torch.cdist(x, cc, compute_mode="donot_use_mm_for_euclid_dist") ** 2
    assert (dist.gather(1, A[:, :1])[:, 0] <= dist.min(1)[0] * (1 + 1e-5)).all()
    r = x - cc[A[:, 0]]
    r = r / r.norm(dim=1, keepdim=True).clamp(min=1e-30)
    loss = dist + 1.5 * ((x * r).sum(1, keepdim=True) - r @ cc.T) ** 2
    loss.scatter_(1, A[:, :1], float("inf"))
    assert (loss.gather(1, A[:, 1:])[:, 0] <= loss.min(1)[0] * (1 + 1e-5)).all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,k", [(80, 10), (88, 10), (80, 11), (88, 16), (96, 16), (104, 10), (104, 16), (144, 12)])
def test_long_partitions_of_either_tile(soar, dtype, d, k):
    """64- and 128-row tiles (k = 10, 88 columns) with every length of the shared candidate lists, tight clusters."""
    g = torch.Generator(device="cuda").manual_seed(d + k)
    n = 70_000
    X = torch.randn(n, d, generator=g, device="cuda")
    X[::3] = X[0] + 0.02 * X[::3]
    X = torch.nn.functional.normalize(X, dim=1).to(dtype)
    Q = torch.nn.functional.normalize(torch.randn(140, d, generator=g, device="cuda"), dim=1)
    Q[::7] = X[0].float() + 0.02 * Q[::7]
    full = Q.double() @ X.double().T
    want = full.topk(k, 1)[0]
    C = X[:4].float().contiguous()
    A = soar.soar_assign(X, C, 1.0, 1)
    ix = soar.soar_index_build(X, C, A)
    for ids, sc in (soar.soar_exact_mips(X, Q, k), soar.soar_search(ix, Q, k, 4)):
        assert torch.allclose(sc.double(), want, rtol=0, atol=1e-5)
        assert torch.allclose(full.gather(1, ids), want, rtol=0, atol=1e-5)
        assert all(ids[q].unique().numel() == k for q in range(0, 140, 20))
    ix.close()


@pytest.mark.parametrize("c", [448, 449, 512, 513])
@pytest.mark.parametrize("nq", [1, 129, 700])
def test_selection_around_the_split(soar, c, nq):
    g = torch.Generator().manual_seed(c)
    C, Q = torch.randn(c, 40, generator=g).cuda(), torch.randn(nq, 40, generator=g).cuda()
    A = torch.arange(c).int()[:, None].contiguous().cuda()
    ix = soar.soar_index_build(C, C, A)
    top, sc = soar.soar_select_partitions(ix, Q, 17, with_scores=True)
    full = Q.double() @ C.double().T
    want = full.topk(17, 1)[0]
    assert torch.allclose(sc.double(), want, rtol=1e-5, atol=1e-4)
    assert torch.allclose(full.gather(1, top.long()), want, rtol=1e-5, atol=1e-4)
    assert all(top[q].unique().numel() == 17 for q in range(nq))
    ix.close()
