"""Tile edges, remainders and rarely taken branches of the GPU kernels, against fp64 references."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d_in,hidden", [(1, 1, 1), (33, 17, 63), (129, 64, 65), (700, 165, 130), (260, 33, 300)])
def test_mlp_gradients_at_tile_edges(soar, B, d_in, hidden):
    g = torch.Generator().manual_seed(B)
    n1, n2 = hidden * d_in, hidden * hidden
    params = 0.3 * torch.randn(soar.soar_mlp_param_count(d_in, hidden), generator=g)
    Z, target = torch.randn(B, d_in, generator=g), torch.randn(B, generator=g)
    G, loss = soar.soar_mlp_backward(params.cuda(), d_in, hidden, Z.cuda(), target.cuda())
    y = soar.soar_mlp_forward(params.cuda(), d_in, hidden, Z.cuda())

    def passes(p, z, t, abs_=False):
        """(y, loss, gradient); with abs_, every term replaced by its magnitude (the scale of the rounding errors)."""
        W1, b1, W2, b2, w3, b3 = torch.split(p, [n1, hidden, n2, hidden, hidden, 1])
        W1, W2 = W1.view(hidden, d_in), W2.view(hidden, hidden)
        a1 = z @ W1.T + b1
        h1 = a1 if abs_ else a1.relu()
        a2 = h1 @ W2.T + b2
        h2 = a2 if abs_ else a2.relu()
        out = h2 @ w3 + b3
        e = out + t if abs_ else out - t
        gy = 2 * e / B
        ga2 = gy[:, None] * w3 * (1 if abs_ else (a2 > 0))
        ga1 = (ga2 @ W2) * (1 if abs_ else (a1 > 0))
        grad = [ga1.T @ z, ga1.sum(0), ga2.T @ h1, ga2.sum(0), gy @ h2, gy.sum()[None]]
        return out, (e * e).mean(), torch.cat([v.reshape(-1) for v in grad])

    p, z, t = params.double(), Z.double(), target.double()
    want = passes(p, z, t)
    scale = passes(p.abs(), z.abs(), t.abs(), True)
    # at most this many roundings lie on the way from an input to a gradient entry
    tol = 2.0 ** -24 * (d_in + 4 * hidden + 2 * B + 40)
    for got, w, s in zip((y, loss[0], G), want, scale):
        assert ((got.cpu().double() - w).abs() <= tol * s).all()


def _index(soar, n, d, c, seed, dtype=torch.float32, copies=0):
    """(X, C, A, index): random unit rows (the first `copies` of them equal) under random rows as centroids."""
    g = torch.Generator().manual_seed(seed)
    X = torch.nn.functional.normalize(torch.randn(n, d, generator=g), dim=1)
    X[:copies] = X[0]
    X = X.to(dtype)
    C = X.float()[torch.randperm(n, generator=g)[:c]].contiguous()
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.0, 1)
    return X, C, A, soar.soar_index_build(X.cuda(), C.cuda(), A)


def _check_search(soar, X, C, A, ix, Q, k, t, tpq=None, sample=40):
    """A sample of the batch against every probed row scored in fp64; an id may differ where scores tie."""
    ids, sc = soar.soar_search(ix, Q.cuda(), k, t, None if tpq is None else tpq.cuda())
    top = soar.soar_select_partitions(ix, Q.cuda(), t).cpu()
    A, Xd = A.cpu(), X.double()
    for q in torch.linspace(0, Q.shape[0] - 1, min(sample, Q.shape[0])).long().tolist():
        m = t if tpq is None else int(tpq[q].clamp(0, t))
        in_union = torch.isin(A, top[q, :m].to(A.dtype)).any(1)
        full = torch.where(in_union, Xd @ Q[q].double(), torch.tensor(-float("inf"), dtype=torch.float64))
        want, at = full.sort(descending=True, stable=True)
        have = min(k, int(in_union.sum()))
        got_i, got_s = ids[q].cpu(), sc[q].cpu().double()
        assert (got_i[have:] == -1).all() and torch.isinf(got_s[have:]).all()
        assert torch.allclose(got_s[:have], want[:have], rtol=0, atol=1e-5)
        assert torch.allclose(full[got_i[:have]], want[:have], rtol=0, atol=1e-5)
        assert got_i[:have].unique().numel() == have


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("nq,k,t,copies", [
    (1, 1, 30, 0),          # one query, one result
    (60, 33, 60, 0),        # smallest k of the wide lists
    (40, 128, 200, 0),      # more lists than a block has threads, largest k
    (50, 100, 60, 700),     # tied rows overflow the lists: rescans by the block
    (50, 10, 60, 700),
    (700, 128, 200, 0), (650, 100, 60, 700),            # narrower blocks: batches of several blocks an SM
    (4200, 10, 4, 700),     # rescans by a warp (large batches)
    (4096, 3, 3, 0), (4097, 3, 3, 0),   # both sides of the block / warp line
])
def test_finishing_of_small_and_wide_searches(soar, dtype, nq, k, t, copies):
    X, C, A, ix = _index(soar, 9000, 24, 260, 3, dtype, copies)
    g = torch.Generator().manual_seed(nq)
    Q = torch.nn.functional.normalize(torch.randn(nq, 24, generator=g), dim=1)
    if copies:
        Q[::2] = X[0].float() + 0.05 * Q[::2]
    tpq = torch.randint(-2, t + 3, (nq,), generator=g).int()     # values outside [0, t] are clamped
    for counts in (None, tpq):
        _check_search(soar, X, C, A, ix, Q, k, t, counts)
    ix.close()


@pytest.mark.parametrize("nq,k", [(20, 20), (20, 128), (620, 40)])
def test_finishing_of_more_lists_than_block_threads(soar, nq, k):
    X, C, A, ix = _index(soar, 9000, 24, 800, 7)
    g = torch.Generator().manual_seed(nq + k)
    Q = torch.nn.functional.normalize(torch.randn(nq, 24, generator=g), dim=1)
    _check_search(soar, X, C, A, ix, Q, k, 700)
    _check_search(soar, X, C, A, ix, Q, k, 700, torch.randint(0, 701, (nq,), generator=g).int())
    ix.close()


@pytest.mark.parametrize("c", [8191, 8192, 9000])
def test_grouping_past_one_scan_block(soar, c):
    X, C, A, ix = _index(soar, 20_000, 16, c, 5)
    g = torch.Generator().manual_seed(c)
    Q = torch.nn.functional.normalize(torch.randn(5000, 16, generator=g), dim=1)
    _check_search(soar, X, C, A, ix, Q, 10, 8)
    _check_search(soar, X, C, A, ix, Q, 10, 8, torch.randint(0, 9, (5000,), generator=g).int())
    ix.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,d,shift", [(7, 5, 0), (8, 8, 0), (9, 8, 1), (1000, 33, 3), (700, 96, 0), (65_541, 24, 1)])
def test_row_copies_of_odd_and_unaligned_rows(soar, dtype, n, d, shift):
    g = torch.Generator().manual_seed(n)
    flat = torch.randn(n * d + shift, generator=g).to(dtype).cuda()
    X = flat[shift:].view(n, d)                                  # rows that need not start on 16 bytes
    Q = torch.randn(37, d, generator=g).cuda()
    c = max(2, n // 50)
    C = X[:c].float().contiguous()
    A = soar.soar_assign(X, C, 1.0, 1)
    ix = soar.soar_index_build(X, C, A)
    rows = ix.vectors()
    assert torch.equal(rows[:, :d], X[ix.ids().long()]) and not rows[:, d:].any()
    k = min(10, n)
    full = Q.double() @ X.double().T
    want = full.topk(k, 1)[0]
    for ids, sc in (soar.soar_search(ix, Q, k, c), soar.soar_exact_mips(X, Q, k)):
        assert torch.allclose(sc.double(), want, rtol=1e-5, atol=1e-4)
        assert torch.allclose(full.gather(1, ids), want, rtol=1e-5, atol=1e-4)
    ix.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,big", [(3, 0.0), (130, 0.0), (130, 2e38)])
def test_centroid_means_of_every_cluster_size(soar, dtype, d, big):
    """Clusters of 1 to 140 rows (every remainder of the summation's batches); `big` makes fp32 sums overflow."""
    g = torch.Generator().manual_seed(d)
    sizes = torch.arange(1, 141)
    c = sizes.numel()
    centre = 1000.0 * torch.arange(1, c + 1)[:, None] * torch.nn.functional.one_hot(torch.arange(c) % d, d)
    own = torch.repeat_interleave(torch.arange(c), sizes)
    X = (centre[own] + torch.randn(own.numel(), d, generator=g)).to(dtype)
    if big:                                        # one more cluster far away whose sums exceed fp32
        far = torch.full((40, d), big).to(dtype)
        X, own, c = torch.cat([X, far]), torch.cat([own, torch.full((40,), c)]), c + 1
    first = torch.tensor([int((own == j).nonzero()[0]) for j in range(c)]).int()
    C = soar.soar_train_centroids(X.cuda(), c, 1, first.cuda()).cpu()
    a = soar.soar_assign(X.cuda(), X.float()[first.long()].contiguous().cuda(), 0.0, 0).cpu()[:, 0].long()
    for j in range(c):
        rows = X[a == j].double()
        if len(rows):
            want = rows.mean(0).float()
            assert ((C[j] - want).abs() <= 2.0 ** -23 * want.abs()).all(), j


def _fp8_rows(V):
    scale = V.abs().amax(1, keepdim=True) / 448
    scale = torch.where(scale > 0, scale, torch.ones_like(scale))
    return (V / scale).to(torch.float8_e4m3fn).double() * scale.double()


@pytest.mark.parametrize("mode", ["fp8", "pq4"])
@pytest.mark.parametrize("d,c,t,R,copies", [
    (16, 60, 3, 1, 0), (34, 60, 4, 33, 0),       # one row kept; lists past a warp
    (300, 60, 4, 100, 0),                        # rows wider than one register fragment
    (24, 300, 250, 100, 0),                      # more earlier probes than the hash table takes
    (24, 60, 6, 700, 3000),                      # thousands of equal scores at the threshold
    (24, 60, 60, 4096, 0),                       # the largest shortlist
])
def test_shortlists_at_their_limits(soar, mode, d, c, t, R, copies):
    g = torch.Generator().manual_seed(d + c)
    n, nq = 8000, 40
    X = torch.nn.functional.normalize(torch.randn(n, d, generator=g), dim=1)
    X[1000:1000 + copies] = X[0]
    Q = torch.nn.functional.normalize(torch.randn(nq, d, generator=g), dim=1)
    if copies:
        Q[::2] = X[0] + 0.3 * Q[::2]
    C = X[torch.randperm(1000, generator=g)[:c]].contiguous()
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.0, 1)
    if mode == "fp8":
        ix = soar.soar_index_build(X.cuda(), C.cuda(), A, mode=soar.SOAR_SCORE_FP8)
        approx = _fp8_rows(Q) @ _fp8_rows(X).T
        approx = approx[:, :, None].expand(-1, -1, 2)
    else:
        B = 0.3 * torch.randn(d // 2, 16, 2, generator=g)
        ix = soar.soar_index_build_pq(X.cuda(), C.cuda(), A, B.cuda())
        copies_hat = []
        for col in range(2):
            base = C[A[:, col].cpu().long()]
            r = (X - base).view(n, -1, 2)
            code = ((r[:, :, None] - B[None]) ** 2).sum(3).argmin(2)
            copies_hat.append(base + B[torch.arange(d // 2)[None], code].reshape(n, d))
        approx = torch.stack([Q.double() @ h.double().T for h in copies_hat], 2)
    top = soar.soar_select_partitions(ix, Q.cuda(), t).cpu().long()
    A = A.cpu().long()
    k = min(R, 1024)
    ids, sc = soar.soar_search(ix, Q.cuda(), k, t, rescore=R)
    full = Q.double() @ X.double().T
    for q in range(nq):
        place = torch.full((c,), 10 ** 6).scatter_(0, top[q], torch.arange(t))
        first = place[A].argmin(1)                                   # the copy in the earliest-probed partition
        s = approx[q].gather(1, first[:, None])[:, 0]
        inside = (place[A] < 10 ** 6).any(1)
        s = torch.where(inside, s, torch.tensor(-float("inf"), dtype=torch.float64))
        order = s.sort(descending=True, stable=True)[1]
        short = order[: min(R, int(inside.sum()))]
        got = ids[q].cpu()
        got = got[got >= 0]
        assert got.unique().numel() == got.numel() == min(k, short.numel())
        # fp32 sums of d products: a score may change places only within this of the R-th
        slack = d * 2.0 ** -21
        assert (s[got] >= s[short[-1]] - slack).all()
        sure = short[s[short] > s[short[-1]] + slack] if short.numel() == R else short
        if sure.numel() == short.numel():
            want = full[q, short].sort(descending=True)[0][:k]
            assert torch.allclose(full[q, got], want, rtol=0, atol=1e-5)
        if k == short.numel():
            assert torch.isin(sure, got).all()
        if copies and q % 2 == 0 and mode == "fp8":                  # equal scores: the lower ids are kept
            tied = s[got] == s[0]
            kept = got[tied].sort()[0]
            all_tied = torch.nonzero(s == s[0])[:, 0]
            assert torch.equal(kept, all_tied[: kept.numel()])
    ix.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,c,n", [(5, 2, 1), (100, 129, 255), (100, 128, 257), (126, 300, 300), (134, 257, 700), (150, 257, 300), (158, 257, 300),
                                   (142, 257, 300), (278, 130, 200), (64, 3000, 513)])
def test_assignment_shapes(soar, dtype, d, c, n):
    """Ragged point blocks and codebook tiles; rows too wide for long stages (126..150) or lists (158) and for two operands (142..278)."""
    g = torch.Generator().manual_seed(d + c)
    X = torch.randn(n, d, generator=g).to(dtype)
    C = torch.randn(c, d, generator=g)
    if c > 2000:                                    # dozens of near-equal centroids to a point: full lists, rescans
        C = C[:40].repeat_interleave(c // 40, 0)
        C = C + 1e-4 * torch.randn(C.shape, generator=g)
    A = soar.soar_assign(X.cuda(), C.cuda(), 1.5, 1).cpu().long()
    x, cc = X.double(), C.double()
    dist = torch.cdist(x, cc, compute_mode="donot_use_mm_for_euclid_dist") ** 2
    first = A[:, 0]
    got = dist.gather(1, first[:, None])[:, 0]
    assert (got <= dist.min(1)[0] * (1 + 1e-5)).all()
    r = x - cc[first]
    r = r / r.norm(dim=1, keepdim=True).clamp(min=1e-30)
    loss = dist + 1.5 * ((x * r).sum(1, keepdim=True) - r @ cc.T) ** 2
    loss.scatter_(1, first[:, None], float("inf"))
    assert (first != A[:, 1]).all()
    assert (loss.gather(1, A[:, 1:])[:, 0] <= loss.min(1)[0] * (1 + 1e-5)).all()


@pytest.mark.parametrize("nq,c,t", [(1, 130, 32), (1, 5300, 7), (129, 700, 17), (300, 9000, 16)])
def test_selection_split_over_the_codebook(soar, nq, c, t):
    """Parts that cut through query blocks, with three equal centroids among them."""
    g = torch.Generator().manual_seed(c)
    C = torch.randn(c, 40, generator=g)
    C[c // 2] = C[c - 1] = C[3]
    X = torch.randn(c, 40, generator=g)
    A = torch.arange(c).int()[:, None].contiguous()
    ix = soar.soar_index_build(X.cuda(), C.cuda(), A.cuda())
    Q = torch.randn(nq, 40, generator=g)
    Q[0] = C[3]
    top, sc = soar.soar_select_partitions(ix, Q.cuda(), t, with_scores=True)
    full = Q.double() @ C.double().T
    want = full.topk(t, 1)[0]
    assert torch.allclose(sc.cpu().double(), want, rtol=1e-5, atol=1e-4)
    assert torch.allclose(full.gather(1, top.cpu().long()), want, rtol=1e-5, atol=1e-4)
    assert all(top[q].unique().numel() == t for q in range(nq))
    assert top[0, :3].tolist() == [3, c // 2, c - 1]          # equal scores: the lower id first
    ix.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("nq,k,t", [(1, 10, 14), (1, 32, 30), (3, 1, 20), (9, 32, 7), (70, 5, 3)])
def test_few_queries_split_partitions_over_warps(soar, dtype, nq, k, t):
    X, C, A, ix = _index(soar, 9000, 24, 110, 7, dtype, copies=50)
    g = torch.Generator().manual_seed(nq)
    Q = torch.nn.functional.normalize(torch.randn(nq, 24, generator=g), dim=1)
    Q[0] = X[0].float()
    for counts in (None, torch.randint(0, t + 1, (nq,), generator=g).int()):
        _check_search(soar, X, C, A, ix, Q, k, t, counts)
    ix.close()


@pytest.mark.parametrize("dtype,d", [(torch.float32, 100), (torch.float32, 130), (torch.bfloat16, 48)])
@pytest.mark.parametrize("n,k", [(65_536 + 64, 10), (65_536 * 2 + 65, 16), (70_001, 1)])
def test_brute_force_over_long_chunks(soar, dtype, d, n, k):
    """Chunks whose last tile holds 64, 65 or a few rows; tight clusters and equal rows near the top."""
    g = torch.Generator(device="cuda").manual_seed(n + d)
    X = torch.randn(n, d, generator=g, device="cuda")
    X[::3] = X[0] + 0.02 * X[::3]
    X = torch.nn.functional.normalize(X, dim=1)
    X[n - 40:] = X[0]
    X = X.to(dtype)
    Q = torch.cat([X[:1].float(), torch.nn.functional.normalize(torch.randn(140, d, generator=g, device="cuda"), dim=1)])
    ids, sc = soar.soar_exact_mips(X, Q, k)
    full = Q.double() @ X.double().T
    want = full.topk(k, 1)[0]
    assert torch.allclose(sc.double(), want, rtol=0, atol=1e-5)
    assert torch.allclose(full.gather(1, ids), want, rtol=0, atol=1e-5)
    assert all(ids[q].unique().numel() == k for q in range(0, 141, 20))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,nq,k", [
    (1, 1, 1), (511, 3, 128), (513, 129, 10),       # one and two chunks of the least size
    (77_825, 1, 16), (77_825, 128, 33),             # 512 rows a chunk on 152 SMs, and one row past them
    (65_537, 20_000, 1), (131_072, 2000, 10),       # longest chunks, several waves
    (131_072, 2000, 17), (131_072, 5000, 32), (20_000, 200, 20), (20_000, 200, 17), (3000, 50, 29), (700, 20, 32),
])
def test_brute_force_chunks_of_every_size(soar, dtype, n, nq, k):
    g = torch.Generator().manual_seed(n + nq)
    X = torch.randn(n, 24, generator=g).to(dtype).cuda()
    Q = torch.randn(nq, 24, generator=g).cuda()
    ids, sc = soar.soar_exact_mips(X, Q, min(k, n))
    at = torch.linspace(0, nq - 1, min(nq, 64)).long().cuda()
    full = Q[at].double() @ X.double().T
    want = full.topk(min(k, n), 1)[0]
    assert torch.allclose(sc[at].double(), want, rtol=1e-5, atol=1e-4)
    assert torch.allclose(full.gather(1, ids[at]), want, rtol=1e-5, atol=1e-4)
