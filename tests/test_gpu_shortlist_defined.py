"""The compressed searches against their definition, bit for bit: the shortlist is the R best approximate scores,
each summed in fp32 in ascending order (score descending, lower id first), and k = R returns all of it.

The tensor cores sum in another order.  Their error has to stay within the bound that the selection allows for it,
which these inputs press: scores that differ by a few roundings, one large product above many small ones, rows of
very uneven length."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fp32_chain(a, b):
    """fp32 sums over the last dimension in ascending order, one rounding a term, of products that 53 bits hold."""
    acc = torch.zeros(torch.broadcast_shapes(a.shape, b.shape)[:-1], dtype=torch.float32, device=a.device)
    for k in range(a.shape[-1]):
        acc = (acc.double() + a[..., k].double() * b[..., k].double()).float()
    return acc


def _fp8_scores(soar, Q, X):
    (xc, xs), (qc, qs) = ([v.cpu() for v in soar.soar_quantize_fp8(V.cuda())] for V in (X, Q))
    xv, qv = (v.view(torch.float8_e4m3fn).float() for v in (xc, qc))
    return _fp32_chain(qv[:, None], xv[None]) * qs[:, None] * xs[None]


def _best(score, ids, count):
    """The ids of the `count` best scores, lower ids first."""
    return ids[torch.sort(score, descending=True, stable=True)[1][:count]]


def _check(soar, ix, c, A, X, Q, score_of_copy, t, R, k):
    """score_of_copy [nq, n, 1 + spills]: the defined score of every copy.  (The reference runs on the CPU.)"""
    top = soar.soar_select_partitions(ix, Q.cuda(), t).cpu().long()
    ids, sc = (v.cpu() for v in soar.soar_search(ix, Q.cuda(), k, t, rescore=R))
    full = Q.double() @ X.double().T
    size = Q.double().abs() @ X.double().abs().T
    for q in range(Q.shape[0]):
        place = torch.full((c,), 10 ** 6).scatter_(0, top[q], torch.arange(t))
        first = place[A].argmin(1)                               # a point counts by its copy probed first
        inside = torch.nonzero((place[A] < 10 ** 6).any(1))[:, 0]    # (ascending ids)
        s = score_of_copy[q].gather(1, first[:, None])[inside, 0]
        short = _best(s, inside, min(R, inside.numel()))
        have = min(k, short.numel())
        got, gs = ids[q, :have], sc[q, :have].double()
        assert (ids[q, have:] == -1).all() and got.unique().numel() == have
        assert torch.isin(got, short).all()
        # the exact scores: fp32 sums of d products
        tol = 2.0 ** -23 * X.shape[1] * size[q]
        assert ((gs - full[q, got]).abs() <= tol[got]).all()
        assert ((gs[1:] < gs[:-1]) | ((gs[1:] == gs[:-1]) & (got[1:] > got[:-1]))).all()
        if have < short.numel():
            left = short[~torch.isin(short, got)]
            assert (full[q, left] <= gs[-1] + tol[left]).all()


def _rows(pattern, n, d, g):
    X = torch.nn.functional.normalize(torch.randn(n, d, generator=g), dim=1)
    if pattern == "outliers":
        X[:: n // 9] *= 1000
    elif pattern == "two_sizes":
        X[::100] *= 1000
    elif pattern == "heavy":
        X *= torch.exp(2 * torch.randn(n, 1, generator=g))
    elif pattern == "ties":
        X[1000:4000] = X[0]
    elif pattern == "one_large":
        # every row's largest code is the first column's; the others shrink over eleven octaves
        X = X * 2.0 ** -torch.randint(0, 12, (n, d), generator=g).float()
        X[:, 0] = 1.0
    return X


@pytest.mark.parametrize("d,R,k", [(24, 100, 100), (96, 1000, 1000), (96, 33, 10), (300, 50, 50), (24, 4096, 1024)])
@pytest.mark.parametrize("pattern", ["even", "outliers", "two_sizes", "heavy", "ties", "one_large"])
def test_fp8_shortlist_is_the_defined_one(soar, pattern, d, R, k):
    g = torch.Generator().manual_seed(d + R)
    n, nq, c, t = 16_000, 12, 40, 12
    X = _rows(pattern, n, d, g)
    Q = torch.nn.functional.normalize(torch.randn(nq, d, generator=g), dim=1)
    if pattern == "one_large":                               # scores that differ by the small products only
        Q[:, 0] = 1.0
        Q[::2, 1:] *= 2.0 ** -8
    if pattern == "ties":
        Q[::2] = X[0] + 0.3 * Q[::2]
    C = torch.nn.functional.normalize(torch.randn(c, d, generator=g), dim=1)
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.0, 1)
    ix = soar.soar_index_build(X.cuda(), C.cuda(), A, mode=soar.SOAR_SCORE_FP8)
    s = _fp8_scores(soar, Q, X)
    _check(soar, ix, c, A.cpu().long(), X, Q, s[:, :, None].expand(-1, -1, 2), t, R, k)
    ix.close()


@pytest.mark.parametrize("d,R,k", [(24, 100, 100), (100, 1000, 1000), (100, 33, 10), (24, 4096, 1024)])
@pytest.mark.parametrize("pattern", ["even", "outliers", "ties", "one_large"])
def test_pq4_shortlist_is_the_defined_one(soar, pattern, d, R, k):
    """Queries, centroids and PQ centres on a grid, so that a term's products are exact and its order fixes the sum."""
    g = torch.Generator().manual_seed(d + R)
    n, nq, c, t = 16_000, 12, 40, 12
    X = _rows(pattern, n, d, g)
    Q = torch.nn.functional.normalize(torch.randn(nq, d, generator=g), dim=1)
    if pattern == "one_large":
        Q[:, 0] = 1.0
    if pattern == "ties":
        Q[::2] = X[0] + 0.3 * Q[::2]
    C = torch.nn.functional.normalize(torch.randn(c, d, generator=g), dim=1)
    Q, C = (torch.round(v * 1024) / 1024 for v in (Q, C))
    B = torch.round(0.3 * torch.randn(d // 2, 16, 2, generator=g) * 256) / 256
    if pattern == "one_large":
        B[0] *= 512
        B[1::2] /= 64
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.0, 1)
    ix = soar.soar_index_build_pq(X.cuda(), C.cuda(), A, B.cuda())
    A = A.cpu().long()
    scores = torch.empty(nq, n, 2)
    m = d // 2
    for col in range(2):
        r = (X - C[A[:, col]]).view(n, m, 1, 2)
        d0, d1 = r[..., 0] - B[None, ..., 0], r[..., 1] - B[None, ..., 1]            # fp32, as the encoder rounds
        code = ((d0 * d0).double() + d1.double() ** 2).float().argmin(2)
        centre = B[torch.arange(m)[None], code]                       # [n, m, 2]
        acc = torch.zeros(nq, n)
        for j in range(m):
            lut = (Q[:, 2 * j + 1].double()[:, None] * centre[:, j, 1].double()
                   + (Q[:, 2 * j, None] * centre[:, j, 0]).double()).float()
            acc = acc + lut
        lanes = torch.zeros(nq, c, 32)
        for k0 in range(0, d, 32):
            w = min(32, d - k0)
            prod = Q[:, None, k0:k0 + w].double() * C[None, :, k0:k0 + w].double()
            lanes[:, :, :w] = (lanes[:, :, :w].double() + prod).float()
        for o in (16, 8, 4, 2, 1):
            lanes = lanes + lanes[:, :, torch.arange(32) ^ o]
        scores[:, :, col] = lanes[:, :, 0][:, A[:, col]] + acc
    _check(soar, ix, c, A, X, Q, scores, t, R, k)
    ix.close()


@pytest.mark.parametrize("n,c,t,spills", [
    (3000, 300, 250, 1), (3000, 300, 250, 2),       # more earlier probes than the largest table, fewer partitions
    (9000, 4000, 900, 2),                           # more of both than the largest table: compared
    (700, 100, 3, 1),                               # fewer rows than the shortlist
])
def test_fp8_shortlist_of_many_probes(soar, n, c, t, spills):
    g = torch.Generator().manual_seed(n)
    d, nq = 24, 12
    X = _rows("even", n, d, g)
    Q = torch.nn.functional.normalize(torch.randn(nq, d, generator=g), dim=1)
    C = X[torch.randperm(n, generator=g)[:c]].contiguous()
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.0, spills)
    ix = soar.soar_index_build(X.cuda(), C.cuda(), A, mode=soar.SOAR_SCORE_FP8)
    s = _fp8_scores(soar, Q, X)
    _check(soar, ix, c, A.cpu().long(), X, Q, s[:, :, None].expand(-1, -1, 1 + spills), t, 200, 200)
    ix.close()


@pytest.mark.parametrize("R", [10, 100])
def test_fp8_shortlist_of_a_long_slice(soar, R):
    """More rows above the sampled floor than are kept: the bins run over the whole slice."""
    g = torch.Generator().manual_seed(R)
    n, d, c, nq = 300_000, 16, 3, 3
    X = torch.nn.functional.normalize(torch.randn(n, d, generator=g), dim=1)
    Q = torch.nn.functional.normalize(torch.randn(nq, d, generator=g), dim=1)
    C = X[:c].contiguous()
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.0, 1)
    ix = soar.soar_index_build(X.cuda(), C.cuda(), A, mode=soar.SOAR_SCORE_FP8)
    s = _fp8_scores(soar, Q, X)
    _check(soar, ix, c, A.cpu().long(), X, Q, s[:, :, None].expand(-1, -1, 2), c, R, R)
    ix.close()
