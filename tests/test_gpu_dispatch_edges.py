"""Kernels that a size rule picks, at the sizes where they can go wrong: the smallest and largest of their range, remainders
of their tiles, and inputs that leave their common path.  Oracle or sibling kernel as the reference, exact where the result is."""
import numpy as np
import pytest
import torch

from oracle import fathom_oracle as O

pytestmark = pytest.mark.gpu


# (tokens, k, sink, local): one CTA and clusters of 2, 4 and 8; 8, 16 and 32 scores per thread; one past each; up to the longest row
@pytest.mark.parametrize("n,k,n_sink,n_local", [(1, 1, 0, 0), (31, 7, 0, 0), (64, 64, 4, 32), (4096, 64, 0, 0), (4097, 1000, 4, 32), (8193, 8193, 0, 0),
                                                (16385, 5, 0, 0), (32768, 2048, 0, 0), (32769, 9000, 4, 32), (65536, 36, 4, 32),
                                                (65537, 512, 0, 0), (131071, 4096, 4, 32), (131072, 16384, 0, 0)])
@pytest.mark.parametrize("scores", ["spread", "ties", "equal", "negative"])
def test_topk_of_rows_held_in_registers(n, k, n_sink, n_local, scores):
    from paper_2609_17652_b200 import binding as fb
    Hq = 3
    lay = fb.make_layout(1, Hq, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    g = torch.Generator(device="cuda").manual_seed(n + k)
    s = torch.randn(Hq, lay.score_stride, generator=g, device="cuda")
    if scores == "ties":
        s = (s * 4).round() * 0.25                                   # some thirty values, zeros of both signs among them
    elif scores == "equal":
        s = torch.full_like(s, -1.5)
    elif scores == "negative":
        s = -torch.exp(12 * s)                                       # magnitudes outside the finely divided octaves
    s[:, n:] = float("nan")
    idx = torch.full((Hq, k), -1, dtype=torch.int32, device="cuda")
    ctx.fathom_topk(lay, s, k, n_sink, n_local, idx)
    ref = O.topk(s[:, :n].double().cpu().numpy(), k, n_sink, n_local)
    assert np.array_equal(idx.cpu().numpy(), ref)
    assert ctx.fathom_device_status() == 0
    ctx.close()


# rows of which one CTA's chunks of 128 tokens hold more than its share: the lists are made a second time with the threshold of the
# first, or do not fit; few and many heads (8, 16 and 32 scores per thread for the same length)
@pytest.mark.parametrize("Hq,n,k,n_sink,n_local", [(2, 20000, 700, 0, 0), (40, 20000, 700, 4, 32), (33, 33001, 2048, 0, 2000), (2, 65536, 4096, 100, 0),
                                                   (20, 131072, 512, 0, 0), (9, 8200, 4000, 0, 0), (20, 20000, 8192, 0, 0)])
@pytest.mark.parametrize("scores", ["one CTA", "one CTA, few", "rising", "end", "infinite"])
def test_topk_of_uneven_rows_held_in_registers(Hq, n, k, n_sink, n_local, scores):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(1, Hq, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    g = torch.Generator(device="cuda").manual_seed(n + k)
    s = torch.randn(Hq, lay.score_stride, generator=g, device="cuda")
    t = torch.arange(lay.score_stride, device="cuda")
    if scores == "one CTA":
        s += 50.0 * (t // 128 % 8 == 3)
    elif scores == "one CTA, few":
        s += 50.0 * ((t // 128 % 8 == 3) & (t % 128 < 5))
    elif scores == "rising":
        s += 1e-3 * t
    elif scores == "end":
        s += 50.0 * (t >= n - n // 16)
    else:
        s = torch.where(t // 128 % 4 == 1, -float("inf") * torch.ones_like(s), s)
        s[:, n // 2:n // 2 + 9] = float("inf")
    s[:, n:] = float("nan")
    idx = torch.full((Hq, k), -1, dtype=torch.int32, device="cuda")
    ctx.fathom_topk(lay, s, k, n_sink, n_local, idx)
    assert np.array_equal(idx.cpu().numpy(), O.topk(s[:, :n].double().cpu().numpy(), k, n_sink, n_local))
    assert ctx.fathom_device_status() == 0
    ctx.close()


# a context sized for one length serves every shorter one, over the lengths at which the selection changes its way
@pytest.mark.parametrize("longest", [131073, 150001])
def test_shorter_sessions_on_a_longer_sessions_context(longest):
    from paper_2609_17652_b200 import binding as fb
    Hq, k = 4, 64
    ctx = fb.Context(0, fb.fathom_scratch_bytes(fb.make_layout(1, Hq, longest), k))
    g = torch.Generator(device="cuda").manual_seed(longest)
    for n in (longest, 131072, 104001, 33001, 64):
        lay = fb.make_layout(1, Hq, n)
        K = torch.randn(1, n, 128, generator=g, device="cuda")
        q = torch.randn(Hq, 128, generator=g, device="cuda")
        planes = torch.zeros(1, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
        scales = torch.zeros(1, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
        depth = torch.zeros(1, 128, dtype=torch.uint8, device="cuda")
        scores = torch.zeros(Hq, lay.score_stride, device="cuda")
        idx, fused = (torch.full((Hq, k), -1, dtype=torch.int32, device="cuda") for _ in range(2))
        ctx.fathom_build_planes(lay, K, planes, scales)
        ctx.fathom_alloc_depth(lay, q, K.var(dim=1), fb.DEPTH_WATERFILL, 48, 4, depth)
        ctx.fathom_scan(lay, planes, scales, q, depth, 4, scores)
        ctx.fathom_topk(lay, scores, k, 0, 0, idx)
        ctx.fathom_scan_topk(lay, planes, scales, q, depth, 4, k, 0, 0, fused)
        assert np.array_equal(idx.cpu().numpy(), O.topk(scores[:, :n].double().cpu().numpy(), k, 0, 0)), n
        assert torch.equal(idx, fused), n
    ctx.close()


# the longest sequence whose bitmap fits in shared memory and one token more; an odd length with picks in its first and last word
@pytest.mark.parametrize("n,k", [(33, 33), (70001, 700), (52 * 1024 * 32, 2048), (52 * 1024 * 32 + 1, 2048)])
def test_union_of_picks_on_both_sides_of_the_bitmap_limit(n, k):
    from paper_2609_17652_b200 import binding as fb
    Hkv, G = 2, 4
    r = np.random.default_rng(n)
    idx = np.stack([np.sort(np.concatenate([[0, n - 1], 1 + r.choice(n - 2, k - 2, replace=False)])) for _ in range(Hkv * G)]).astype(np.int32)
    lay = fb.make_layout(Hkv, Hkv * G, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    K = torch.randn(Hkv, n, 128, device="cuda").to(torch.bfloat16)
    Ks, Vs = (torch.zeros(Hkv, G * k, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    local = torch.full((Hkv * G, k), -1, dtype=torch.int32, device="cuda")
    count = torch.zeros(Hkv, dtype=torch.int32, device="cuda")
    ctx.fathom_gather_union(lay, torch.from_numpy(idx).cuda(), k, K, K, Ks, Vs, local, count)
    for h in range(Hkv):
        tokens = np.unique(idx[h * G:(h + 1) * G])
        assert int(count[h]) == len(tokens)
        assert np.array_equal(tokens[local[h * G:(h + 1) * G].cpu().numpy()], idx[h * G:(h + 1) * G])
        rows = K[h][torch.from_numpy(tokens.astype(np.int64)).cuda()]
        assert torch.equal(Ks[h, :len(tokens)], rows) and torch.equal(Vs[h, :len(tokens)], rows)
    ctx.close()


# one CTA and clusters of 2 and 8; 4 and 8 rows per half-warp; full and ragged last CTAs; the last k of the small kernel and one more
@pytest.mark.parametrize("k", [1, 3, 64, 65, 511, 512, 513, 1023, 1024, 1025])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_attention_over_few_rows(k, dtype):
    from paper_2609_17652_b200 import binding as fb
    n, Hkv, Hq = 3001, 2, 6
    lay = fb.make_layout(Hkv, Hq, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    g = torch.Generator(device="cuda").manual_seed(k)
    q = 2.0 * torch.randn(Hq, 128, generator=g, device="cuda")
    K, V = (torch.randn(Hkv, n, 128, generator=g, device="cuda").to(dtype) for _ in range(2))
    idx = torch.stack([torch.randperm(n, generator=g, device="cuda")[:k].sort().values for _ in range(Hq)]).to(torch.int32)
    out = torch.full((Hq, 128), float("nan"), device="cuda")
    ctx.fathom_sparse_attend(lay, q, K, V, idx, k, 1.0 / np.sqrt(128), out)
    ref = O.sparse_attend(q.cpu().numpy(), K.float().cpu().numpy(), V.float().cpu().numpy(), idx.cpu().numpy(), 1.0 / np.sqrt(128))
    # logits below 12 in magnitude, each an fp32 sum of 128 products: their rounding, exponentiated, stays below 1e-5
    assert np.all(np.linalg.norm(out.cpu().numpy() - ref, axis=1) <= 2e-5 * np.linalg.norm(ref, axis=1))
    ctx.close()


# every kernel of the chain may start while the one before it still writes; the buffers between them hold the step before's results
def test_dependent_kernels_read_what_the_kernel_before_them_wrote():
    from paper_2609_17652_b200 import binding as fb
    n, Hkv, G, k, steps = 5003, 2, 4, 300, 12
    Hq = Hkv * G
    lay, staged = fb.make_layout(Hkv, Hq, n), fb.make_layout(Hkv, Hq, G * k)
    ctx = fb.Context(0, max(fb.fathom_scratch_bytes(lay, k), fb.fathom_scratch_bytes(staged, k)))
    g = torch.Generator(device="cuda").manual_seed(7)
    K, V = (torch.randn(Hkv, n, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    # early steps take few distinct tokens, late ones many: a length or a list of the step before would show
    scores = [torch.randn(Hq, lay.score_stride, generator=g, device="cuda") * t / steps for t in range(steps)]
    shared = torch.randn(Hkv, 1, lay.score_stride, generator=g, device="cuda").expand(-1, G, -1).reshape(Hq, -1)
    q = [torch.randn(Hq, 128, generator=g, device="cuda") for _ in range(steps)]
    Ks, Vs = (torch.zeros(Hkv, G * k, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx, local = (torch.zeros(Hq, k, dtype=torch.int32, device="cuda") for _ in range(2))
    count, out = torch.zeros(Hkv, dtype=torch.int32, device="cuda"), torch.zeros(Hq, 128, device="cuda")
    rows = [(shared + s).contiguous() for s in scores]
    torch.cuda.synchronize()
    seen = []
    for s, x in zip(rows, q):
        ctx.fathom_topk(lay, s, k, 0, 0, idx)
        ctx.fathom_gather_union(lay, idx, k, K, V, Ks, Vs, local, count)
        ctx.fathom_sparse_attend(staged, x, Ks, Vs, local, k, 1.0 / np.sqrt(128), out)
        seen.append([t.clone() for t in (idx, local, count, out)])
    for s, x, (i, l, c, o) in zip(rows, q, seen):
        ref = O.topk(s[:, :n].double().cpu().numpy(), k, 0, 0)
        assert np.array_equal(i.cpu().numpy(), ref)
        for h in range(Hkv):
            tokens = np.unique(ref[h * G:(h + 1) * G])
            assert int(c[h]) == len(tokens) and np.array_equal(tokens[l[h * G:(h + 1) * G].cpu().numpy()], ref[h * G:(h + 1) * G])
        exact = O.sparse_attend(x.cpu().numpy(), K.float().cpu().numpy(), V.float().cpu().numpy(), ref, 1.0 / np.sqrt(128))
        # logits below 6 in magnitude, fp32 sums of 128 products
        assert np.all(np.linalg.norm(o.cpu().numpy() - exact, axis=1) <= 2e-5 * np.linalg.norm(exact, axis=1))
    ctx.close()


# limits on both sides of the point from which a wait sleeps between polls; part of the warp gives up before the rest
@pytest.mark.parametrize("tries", [1, 64, 66, 4096])
def test_a_warp_agrees_that_its_wait_ran_out(tries):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(1, 1, 300)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, 64))
    ctx.fathom_selftest_wait_expiry(tries)
    assert ctx.fathom_device_status() == fb.DEV_WAIT_EXPIRED
    K = torch.randn(1, 300, 128, device="cuda")
    out = torch.zeros_like(K)
    ctx.fathom_rotate_keys(lay, K, torch.zeros(1, 128, device="cuda"), torch.eye(128, device="cuda").unsqueeze(0).contiguous(), out)
    # the identity moves no key: what is left out of head and tail of both operands is below 2^-21 of it
    assert ctx.fathom_device_status() == 0 and torch.allclose(out, K, rtol=2.0 ** -21, atol=1e-9)
    ctx.close()


# the basis may replace the covariance: finished in fp64 rounds, and by the sweeps that go on where eigenvalues are close
@pytest.mark.parametrize("spread", [100.0, 1e-5])
def test_klt_basis_in_place(spread):
    from paper_2609_17652_b200 import binding as fb
    kv = 3
    lay = fb.make_layout(kv, kv, 1000)
    ctx = fb.Context(0, 0)
    g = torch.Generator(device="cuda").manual_seed(3)
    Q = torch.linalg.qr(torch.randn(kv, 128, 128, generator=g, device="cuda").double())[0]
    cov = ((Q * (1.0 + spread * torch.linspace(0, 1, 128, device="cuda").double())) @ Q.transpose(1, 2)).float()
    cov = (0.5 * (cov + cov.transpose(1, 2))).contiguous()
    basis, eig = torch.zeros_like(cov), torch.zeros(kv, 128, device="cuda")
    ctx.fathom_klt_basis(lay, cov, basis, eig)
    again, eig_again = cov.clone(), torch.zeros_like(eig)
    ctx.fathom_klt_basis(lay, again, again, eig_again)
    assert torch.equal(again, basis) and torch.equal(eig_again, eig)
    B = basis.double()
    # directions are rounded to fp32 (where fp64 sweeps go on they apply their rotations in fp32: 2e-6 measured)
    assert (B.transpose(1, 2) @ B - torch.eye(128, device="cuda").double()).norm() / np.sqrt(128 * kv) < 1e-5
    ctx.close()


# (tokens, heads, k, 36 of them forced) on both sides of every line between the kernels of the selection, scores that exist and scores that do not: the
# longest row in registers; heads for large, middling and small k; 1, 2, 4 and 8 CTAs of 8, 16 and 32 scores per thread, by lists and without; lists of two
# sevenths of a row, of 9000, and of CTAs that cannot share an SM
@pytest.mark.parametrize("n,Hq,k", [(131072, 2, 16384), (131073, 2, 16384), (65536, 149, 1100), (65537, 55, 4133), (65537, 56, 4133), (131072, 37, 2085), (131072, 38, 2085),
                                    (65537, 129, 1061), (65537, 130, 1061), (65537, 130, 1060), (8000, 80, 300), (8000, 80, 8000), (16000, 40, 300), (16000, 40, 9000),
                                    (30000, 14, 300), (30000, 14, 12000), (16000, 80, 300), (30000, 40, 300), (30000, 40, 12000), (60000, 14, 300), (60000, 14, 16000),
                                    (4096, 3, 1206), (4096, 3, 1207), (131072, 2, 9036), (131072, 2, 9037), (33001, 40, 4700), (33001, 40, 5200),
                                    (16384, 96, 16384), (16384, 128, 12000), (8769, 148, 8769), (16384, 149, 12000)])
def test_selection_on_both_sides_of_its_lines(n, Hq, k):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(1, Hq, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    g = torch.Generator(device="cuda").manual_seed(n + Hq + k)
    K, q = torch.randn(1, n, 128, generator=g, device="cuda"), torch.randn(Hq, 128, generator=g, device="cuda")
    planes = torch.zeros(1, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
    scales = torch.zeros(1, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
    depth, scores = torch.zeros(Hq, 128, dtype=torch.uint8, device="cuda"), torch.zeros(Hq, lay.score_stride, device="cuda")
    idx, fused = (torch.full((Hq, k), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.fathom_build_planes(lay, K, planes, scales)
    ctx.fathom_alloc_depth(lay, q, K.var(dim=1), fb.DEPTH_WATERFILL, 16, 1, depth)
    ctx.fathom_scan(lay, planes, scales, q, depth, 1, scores)
    ctx.fathom_topk(lay, scores, k, 4, 32, idx)
    ctx.fathom_scan_topk(lay, planes, scales, q, depth, 1, k, 4, 32, fused)
    assert np.array_equal(idx.cpu().numpy(), O.topk(scores[:, :n].double().cpu().numpy(), k, 4, 32))
    assert torch.equal(idx, fused) and ctx.fathom_device_status() == 0
    ctx.close()


# statistics on both sides of the lines between their merges: 1, 64 and 65 tiles, few and many KV heads
@pytest.mark.parametrize("kv,n", [(1, 3), (1, 1025), (4, 65536), (5, 65537), (9, 2000)])
def test_statistics_merges(kv, n):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(kv, kv, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, 1))
    g = torch.Generator(device="cuda").manual_seed(n)
    K = 2.0 * torch.randn(kv, n, 128, generator=g, device="cuda") + torch.randn(kv, 1, 128, generator=g, device="cuda")
    mean, var, m2 = (torch.zeros(kv, 128, device="cuda") for _ in range(3))
    cov = torch.zeros(kv, 128, 128, device="cuda")
    ctx.fathom_channel_variance(lay, K, mean, var)
    ctx.fathom_calibrate(lay, K, m2, cov)
    X = K.double()
    mu = X.mean(dim=1)
    C = (X - mu.unsqueeze(1)).transpose(1, 2) @ (X - mu.unsqueeze(1)) / (n - 1)
    v = torch.diagonal(C, dim1=1, dim2=2)
    # variances: fp32 sums of 1024 tokens.  Covariances: an accumulator takes up to 65536 / 29 tokens, eight a step, and every step
    # may round towards zero by 2^-23 of it: up to 283 * 2^-23 = 3.4e-5 (1.1e-5 measured)
    assert (mean - mu).norm() < 1e-6 * mu.norm() and (m2 - mu).norm() < 1e-6 * mu.norm()
    assert (var - v).norm() < 1e-5 * v.norm() and (cov - C).norm() < 5e-5 * C.norm()
    ctx.close()


# picks on both sides of the line between one CTA per KV head and the whole chip
@pytest.mark.parametrize("n,k", [(20000, 1102), (20000, 1103), (70001, 4000)])
def test_union_of_many_picks(n, k):
    from paper_2609_17652_b200 import binding as fb
    Hkv, G = 2, 4
    r = np.random.default_rng(k)
    idx = np.stack([np.sort(r.choice(n, k, replace=False)) for _ in range(Hkv * G)]).astype(np.int32)
    lay = fb.make_layout(Hkv, Hkv * G, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    K = torch.randn(Hkv, n, 128, device="cuda")
    Ks, Vs = (torch.zeros(Hkv, G * k, 128, device="cuda") for _ in range(2))
    local = torch.full((Hkv * G, k), -1, dtype=torch.int32, device="cuda")
    count = torch.zeros(Hkv, dtype=torch.int32, device="cuda")
    ctx.fathom_gather_union(lay, torch.from_numpy(idx).cuda(), k, K, K, Ks, Vs, local, count)
    for h in range(Hkv):
        tokens = np.unique(idx[h * G:(h + 1) * G])
        assert int(count[h]) == len(tokens)
        assert np.array_equal(tokens[local[h * G:(h + 1) * G].cpu().numpy()], idx[h * G:(h + 1) * G])
        rows = K[h][torch.from_numpy(tokens.astype(np.int64)).cuda()]
        assert torch.equal(Ks[h, :len(tokens)], rows) and torch.equal(Vs[h, :len(tokens)], rows)
    ctx.close()


# one plan, fewer CTAs than SMs, more
@pytest.mark.parametrize("plans", [1, 18, 19, 74, 75])
@pytest.mark.parametrize("mode,budget", [("waterfill", 48), ("fixed_top_r", 16), ("uniform", 2)])
def test_depths_of_few_and_many_plans(plans, mode, budget):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(1, plans, 100)
    ctx = fb.Context(0, 0)
    g = torch.Generator(device="cuda").manual_seed(plans)
    q, var = torch.randn(plans, 128, generator=g, device="cuda"), torch.rand(1, 128, generator=g, device="cuda")
    depth = torch.full((plans, 128), 9, dtype=torch.uint8, device="cuda")
    code = dict(waterfill=fb.DEPTH_WATERFILL, fixed_top_r=fb.DEPTH_FIXED_TOP_R, uniform=fb.DEPTH_UNIFORM)[mode]
    ctx.fathom_alloc_depth(lay, q, var, code, budget, 1, depth)
    ref = O.alloc_depth(q.cpu().numpy(), var.cpu().numpy(), mode, budget, 1)
    assert np.array_equal(depth.cpu().numpy(), ref)
    ctx.close()


# one CTA per plan: its candidate lists run over (1200 of them for 512, 256 and 128 places a head)
@pytest.mark.parametrize("heads_per_plan", [1, 2, 4])
def test_fused_selection_with_more_candidates_than_a_cta_lists(heads_per_plan):
    from paper_2609_17652_b200 import binding as fb
    n, Hq, k = 140001, 4, 1200
    lay = fb.make_layout(1, Hq, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    g = torch.Generator(device="cuda").manual_seed(heads_per_plan)
    K, q = torch.randn(1, n, 128, generator=g, device="cuda"), torch.randn(Hq, 128, generator=g, device="cuda")
    planes = torch.zeros(1, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
    scales = torch.zeros(1, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
    depth = torch.zeros(Hq // heads_per_plan, 128, dtype=torch.uint8, device="cuda")
    scores = torch.zeros(Hq, lay.score_stride, device="cuda")
    fused = torch.full((Hq, k), -1, dtype=torch.int32, device="cuda")
    ctx.fathom_build_planes(lay, K, planes, scales)
    ctx.fathom_alloc_depth(lay, q, K.var(dim=1), fb.DEPTH_WATERFILL, 32, heads_per_plan, depth)
    ctx.fathom_scan(lay, planes, scales, q, depth, heads_per_plan, scores)
    fb.fathom_scan_set_ctas_per_plan(1)
    try:
        ctx.fathom_scan_topk(lay, planes, scales, q, depth, heads_per_plan, k, 4, 32, fused)
    finally:
        fb.fathom_scan_set_ctas_per_plan(0)
    assert np.array_equal(fused.cpu().numpy(), O.topk(scores[:, :n].double().cpu().numpy(), k, 4, 32))
    assert ctx.fathom_device_status() == 0
    ctx.close()


# keys alike over runs: samples of whole tiles miss some heads' largest scores, and those heads alone are scanned again; with and without scores that exist
@pytest.mark.parametrize("run", [32, 1024])
@pytest.mark.parametrize("n,k,heads_per_plan", [(140001, 300, 4), (140001, 1000, 1), (300032, 4096, 2)])
def test_selection_where_some_heads_samples_miss(n, k, heads_per_plan, run):
    from paper_2609_17652_b200 import binding as fb
    Hkv, Hq = 2, 8
    lay = fb.make_layout(Hkv, Hq, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, k))
    g = torch.Generator(device="cuda").manual_seed(run + k)
    K, q = torch.randn(Hkv, n, 128, generator=g, device="cuda"), torch.randn(Hq, 128, generator=g, device="cuda")
    K[0] = 0.3 * K[0] + torch.randn(n // run + 1, 128, generator=g, device="cuda").repeat_interleave(run, dim=0)[:n]
    planes = torch.zeros(Hkv, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
    scales = torch.zeros(Hkv, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
    depth = torch.zeros(Hq // heads_per_plan, 128, dtype=torch.uint8, device="cuda")
    scores = torch.zeros(Hq, lay.score_stride, device="cuda")
    idx, fused = (torch.full((Hq, k), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.fathom_build_planes(lay, K, planes, scales)
    ctx.fathom_alloc_depth(lay, q, K.var(dim=1), fb.DEPTH_WATERFILL, 48, heads_per_plan, depth)
    ctx.fathom_scan(lay, planes, scales, q, depth, heads_per_plan, scores)
    ctx.fathom_topk(lay, scores, k, 4, 32, idx)
    ctx.fathom_scan_topk(lay, planes, scales, q, depth, heads_per_plan, k, 4, 32, fused)
    assert np.array_equal(idx.cpu().numpy(), O.topk(scores[:, :n].double().cpu().numpy(), k, 4, 32))
    assert torch.equal(idx, fused) and ctx.fathom_device_status() == 0
    ctx.close()


# block maxima whose eighth is rounded to a subnormal fp16 (quotients of up to 12 steps), to the smallest one and to zero; one block per CTA and eight
@pytest.mark.parametrize("n", [200, 40003])
def test_planes_of_keys_with_subnormal_scales(n):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(1, 1, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, 1))
    g = torch.Generator(device="cuda").manual_seed(n)
    K = torch.randn(1, n, 128, generator=g, device="cuda") * torch.exp2(torch.linspace(-26, -12, 128, device="cuda"))
    planes = torch.zeros(1, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
    scales = torch.zeros(1, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
    ctx.fathom_build_planes(lay, K, planes, scales)
    ref_planes, ref_scales = O.build_planes(K.cpu().numpy())
    nb = ref_planes.shape[-1]
    assert (ref_scales.view(np.uint16) == 0).any() and (ref_scales.view(np.uint16) == 1).any()
    assert np.array_equal(scales[..., :nb].cpu().numpy().view(np.uint16), ref_scales.view(np.uint16))
    assert np.array_equal(planes[..., :nb].cpu().numpy().view(np.uint64), ref_planes)
    # the rotation's own quantiser, against the same keys rotated first: the bits are the same
    V = torch.linalg.qr(torch.randn(1, 128, 128, generator=g, device="cuda"))[0].contiguous()
    mean, rotated = torch.zeros(1, 128, device="cuda"), torch.zeros_like(K)
    again, scales_again = torch.zeros_like(planes), torch.zeros_like(scales)
    ctx.fathom_rotate_keys(lay, K, mean, V, rotated)
    ctx.fathom_build_planes(lay, rotated, planes, scales)
    ctx.fathom_build_planes_rotated(lay, K, mean, V, again, scales_again)
    assert torch.equal(again, planes) and torch.equal(scales_again, scales)
    ctx.close()


# one channel far above the others in every key, bases that mix it in and one that leaves it alone
@pytest.mark.parametrize("far", [1e3, 1e5])
@pytest.mark.parametrize("basis", ["random", "identity"])
def test_rotation_of_keys_with_one_large_channel(far, basis):
    from paper_2609_17652_b200 import binding as fb
    n = 1000
    lay = fb.make_layout(1, 1, n)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, 1))
    g = torch.Generator(device="cuda").manual_seed(int(far))
    K = torch.randn(1, n, 128, generator=g, device="cuda")
    K[..., 5] *= far
    V = torch.eye(128, device="cuda").unsqueeze(0).contiguous() if basis == "identity" else torch.linalg.qr(torch.randn(1, 128, 128, generator=g, device="cuda"))[0].contiguous()
    mean, out = torch.randn(1, 128, generator=g, device="cuda"), torch.zeros_like(K)
    ctx.fathom_rotate_keys(lay, K, mean, V, out)
    X = K.double() - mean.double()
    magnitude = X.abs() @ V.double().abs()
    # the difference from the mean rounded to fp32, three terms of 2^-22 for the parts that are left out, 24 accumulations of up to 2^-23
    # each; 2^-39 of the largest for small elements
    bound = (2.0 ** -24 + 3 * 2.0 ** -22 + 24 * 2.0 ** -23) * magnitude + 2.0 ** -39 * X.abs().amax(dim=2, keepdim=True) * V.double().abs().sum(dim=1, keepdim=True)
    assert ((out.double() - X @ V.double()).abs() <= bound).all() and ctx.fathom_device_status() == 0
    ctx.close()


# importances that are zero, equal, powers of four apart, and at the ends of what fp32 queries and variances give: every tie is decided by
# channel and plane
@pytest.mark.parametrize("budget", [0, 1, 5, 47, 130, 300, 509, 512, 600])
@pytest.mark.parametrize("kind", ["zeros", "ties", "powers", "extremes"])
def test_depths_of_tied_and_extreme_importances(kind, budget):
    from paper_2609_17652_b200 import binding as fb
    Hq, hpp = 4, 2
    lay = fb.make_layout(1, Hq, 64)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, 1))
    rng = np.random.default_rng(budget)
    q = np.ones((Hq, 128), np.float32)
    if kind == "zeros":
        var = np.where(rng.random(128) < 0.6, 0.0, rng.random(128))
    elif kind == "ties":
        var = rng.integers(1, 4, 128).astype(np.float64)
    elif kind == "powers":
        var = 4.0 ** rng.integers(-3, 4, 128) * rng.choice([1.0, 1.0, 2.0], 128)
    else:
        q *= rng.choice(np.array([1e-45, 1e-20, 1.0, 3.4e38], np.float32), (1, 128))
        var = rng.choice([0.0, 1e-45, 1e-30, 1.0, 3.4e38], 128)
    var = var.astype(np.float32)[None]
    depth = torch.full((Hq // hpp, 128), 9, dtype=torch.uint8, device="cuda")
    ctx.fathom_alloc_depth(lay, torch.from_numpy(q).cuda(), torch.from_numpy(var).cuda(), fb.DEPTH_WATERFILL, budget, hpp, depth)
    assert np.array_equal(depth.cpu().numpy(), O.alloc_depth(q, var, "waterfill", budget, hpp))
    ctx.close()


# infinite importances, and ones that are no number (an infinite query times no variance): before all others, one channel after the other
@pytest.mark.parametrize("budget", [1, 4, 6, 17, 60, 300, 512])
@pytest.mark.parametrize("kind", ["infinite", "no number"])
def test_depths_of_importances_that_are_not_finite(kind, budget):
    from paper_2609_17652_b200 import binding as fb
    lay = fb.make_layout(1, 2, 64)
    ctx = fb.Context(0, fb.fathom_scratch_bytes(lay, 1))
    rng = np.random.default_rng(budget)
    q, var = rng.standard_normal((2, 128)).astype(np.float32), rng.random((1, 128)).astype(np.float32)
    far = np.sort(rng.choice(128, 12, replace=False))                # channels of an infinite query; among them some of no variance
    q[0, far[1:]], var[0, far[0]], q[1, 127 - far[0]] = np.inf, np.inf, 3.4e38
    odd = far[2:9:3] if kind == "no number" else far[:0]
    var[0, odd] = 0.0
    var[0, (far[-1] + 1) % 128] = 0.0
    depth = torch.full((1, 128), 9, dtype=torch.uint8, device="cuda")
    ctx.fathom_alloc_depth(lay, torch.from_numpy(q).cuda(), torch.from_numpy(var).cuda(), fb.DEPTH_WATERFILL, budget, 2, depth)
    with np.errstate(invalid="ignore"):
        g = O.importance(q, var, 2)[0]
    assert np.array_equal(np.flatnonzero(np.isnan(g)), odd) and np.isinf(g).any()
    ref, left = np.zeros(128, np.uint8), budget
    for j in odd:
        ref[j] = min(4, left)
        left -= int(ref[j])
    rest = np.setdiff1d(np.arange(128), odd)
    ref[rest] = O.waterfill_depths(g[rest], left)
    assert np.array_equal(depth.cpu().numpy()[0], ref)
    # channels by the sum of magnitudes
    q[1, odd] = np.nan
    ctx.fathom_alloc_depth(lay, torch.from_numpy(q).cuda(), None, fb.DEPTH_FIXED_TOP_R, min(budget, 128), 2, depth)
    w = np.abs(q.astype(np.float64)).sum(axis=0)
    first = sorted(range(128), key=lambda j: (not np.isnan(w[j]), 0.0 if np.isnan(w[j]) else -w[j], j))[:min(budget, 128)]
    assert np.array_equal(np.flatnonzero(depth.cpu().numpy()[0] == 4), np.sort(first)) and set(np.unique(depth.cpu().numpy())) <= {0, 4}
    ctx.close()


# rows at the edges of a stage (16 each; 96 of a tile, 160 of half a tile), half tiles alone on their SMs, whole tiles, half tiles over several waves; tails
# of a block and of a unit
@pytest.mark.parametrize("rows", [15, 17, 96, 97, 113, 144, 159, 160, 161, 255])
@pytest.mark.parametrize("Hkv,n", [(1, 40), (1, 1100), (2, 9000), (2, 33001)])
def test_scan_rows_and_units(Hkv, n, rows):
    from paper_2609_17652_b200 import binding as fb
    from tests._pipeline import score_tolerance
    Hq, hpp = 4 * Hkv, 4
    lay = fb.make_layout(Hkv, Hq, n)
    ctx = fb.Context(0, 0)
    g = torch.Generator(device="cuda").manual_seed(rows)
    K = torch.randn(Hkv, n, 128, generator=g, device="cuda") * torch.exp(2 * torch.rand(Hkv, 1, 128, generator=g, device="cuda"))
    q = torch.randn(Hq, 128, generator=g, device="cuda")
    planes = torch.zeros(Hkv, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
    scales = torch.zeros(Hkv, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
    depth = torch.zeros(Hkv, 128, dtype=torch.uint8, device="cuda")
    scores, walked = (torch.full((Hq, lay.score_stride), -7.0, device="cuda") for _ in range(2))
    ctx.fathom_build_planes(lay, K, planes, scales)
    ctx.fathom_alloc_depth(lay, q, K.var(dim=1), fb.DEPTH_WATERFILL, rows, hpp, depth)
    assert (depth.sum(dim=1) == rows).all()
    ctx.fathom_scan(lay, planes, scales, q, depth, hpp, scores)
    fb.fathom_scan_set_ctas_per_plan(2)                              # whole tiles, several per CTA
    try:
        ctx.fathom_scan(lay, planes, scales, q, depth, hpp, walked)
    finally:
        fb.fathom_scan_set_ctas_per_plan(0)
    assert torch.equal(scores, walked) and (scores[:, n:] == -7.0).all()
    m = min(n, 1100)                                                 # the oracle's share: the first blocks
    nb = (m + 63) // 64
    ref = O.scan(planes[..., :nb].cpu().numpy().view(np.uint64), scales[..., :nb].cpu().numpy().view(np.float16), q.cpu().numpy(), depth.cpu().numpy(), m, hpp)
    assert np.all(np.abs(scores[:, :m].cpu().numpy() - ref) <= score_tolerance(ref))
    ctx.close()


# half tiles over several waves of CTAs give what whole tiles give
@pytest.mark.parametrize("n", [100001, 262144])
@pytest.mark.parametrize("budget", [16, 48, 136])
def test_scan_of_half_tiles_over_waves(n, budget):
    from paper_2609_17652_b200 import binding as fb
    Hkv, Hq, hpp = 8, 16, 2
    lay = fb.make_layout(Hkv, Hq, n)
    ctx = fb.Context(0, 0)
    g = torch.Generator(device="cuda").manual_seed(budget)
    q, var = torch.randn(Hq, 128, generator=g, device="cuda"), torch.rand(Hkv, 128, generator=g, device="cuda")
    planes = torch.randint(-2 ** 62, 2 ** 62, (Hkv, 128, 4, lay.plane_stride_words), generator=g, device="cuda")
    scales = torch.rand(Hkv, 128, lay.scale_stride, generator=g, device="cuda").half().view(torch.int16)
    depth = torch.zeros(Hkv, 128, dtype=torch.uint8, device="cuda")
    scores, walked = (torch.full((Hq, lay.score_stride), -7.0, device="cuda") for _ in range(2))
    ctx.fathom_alloc_depth(lay, q, var, fb.DEPTH_WATERFILL, budget, hpp, depth)
    ctx.fathom_scan(lay, planes, scales, q, depth, hpp, scores)
    fb.fathom_scan_set_ctas_per_plan(30)
    try:
        ctx.fathom_scan(lay, planes, scales, q, depth, hpp, walked)
    finally:
        fb.fathom_scan_set_ctas_per_plan(0)
    assert torch.equal(scores, walked) and (scores[:, n:] == -7.0).all()
    ctx.close()


# plans that fit one stage of half tiles only, and deeper ones: over the host link, and in a batch whose sessions end in a first half or in a second one,
# with CTAs that cross from one session to the next
@pytest.mark.parametrize("budget", [97, 136, 160, 161])
@pytest.mark.parametrize("host,ctas", [(False, None), (False, 3), (True, None)])
def test_deep_plans_of_several_sessions(budget, host, ctas):
    from paper_2609_17652_b200 import binding as fb
    from tests._pipeline import score_tolerance
    Hkv, Hq, hpp = 2, 8, 4
    ctx = fb.Context(0, 0)
    g = torch.Generator(device="cuda").manual_seed(budget)
    items, alone = [], []
    for n in (3000, 512, 4609, 64, 1536, 40):
        lay = fb.make_layout(Hkv, Hq, n)
        q, var = torch.randn(Hq, 128, generator=g, device="cuda"), torch.rand(Hkv, 128, generator=g, device="cuda")
        K = torch.randn(Hkv, n, 128, generator=g, device="cuda")
        planes = torch.zeros(Hkv, 128, 4, lay.plane_stride_words, dtype=torch.int64, device="cuda")
        scales = torch.zeros(Hkv, 128, lay.scale_stride, dtype=torch.int16, device="cuda")
        depth = torch.zeros(Hkv, 128, dtype=torch.uint8, device="cuda")
        scores, single = (torch.full((Hq, lay.score_stride), -7.0, device="cuda") for _ in range(2))
        ctx.fathom_build_planes(lay, K, planes, scales)
        ctx.fathom_alloc_depth(lay, q, var, fb.DEPTH_WATERFILL, budget, hpp, depth)
        ctx.fathom_scan(lay, planes, scales, q, depth, hpp, single)
        if host:
            planes, scales = (torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (planes, scales))
            again = torch.full_like(single, -7.0)
            ctx.fathom_scan(lay, planes, scales, q, depth, hpp, again)
            assert torch.equal(again, single), n
        items.append((lay, planes, scales, q, depth, scores))
        alone.append(single)
    fb.fathom_scan_set_ctas_per_plan(ctas or 0)
    try:
        ctx.fathom_scan_batch(items, hpp)
    finally:
        fb.fathom_scan_set_ctas_per_plan(0)
    for (lay, planes, scales, q, depth, scores), single in zip(items, alone):
        assert torch.equal(scores, single), lay.n
        planes, scales, n = planes.cpu().numpy(), scales.cpu().numpy(), lay.n
        nb = (n + 63) // 64
        ref = O.scan(planes[..., :nb].view(np.uint64), scales[..., :nb].view(np.float16), q.cpu().numpy(), depth.cpu().numpy(), n, hpp)
        assert np.all(np.abs(scores[:, :n].cpu().numpy() - ref) <= score_tolerance(ref))
    ctx.close()
