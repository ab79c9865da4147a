"""Each path of the operators' dispatch at the sizes where it can go wrong (edges of tiles, groups and
cluster sizes, the smallest and largest of a range, general alignments) against fp64."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ats():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2410_05165_gb300 as m
    return m


def _randn(shape, seed, std=1.0, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) * std).to(dtype)


def _x(T, K, seed):
    """T token rows in the padded buffer the GEMMs want; the padding holds NaN (it must not matter)."""
    X = torch.full(((T + 255) // 256 * 256, K), float("nan"), device="cuda", dtype=torch.bfloat16)
    X[:T] = _randn((T, K), seed)
    return X


# M: one partial tile up to several; K: one k-block (clusters of one), few, many; T: group, round and
# token-tile edges
GEMM = [(1, 64, 1), (127, 64, 16), (129, 128, 17), (300, 192, 31), (128, 448, 32), (640, 512, 33), (2304, 768, 64),
        (1920, 1024, 65), (1000, 2048, 127), (4096, 1024, 128), (768, 4096, 129), (3000, 640, 250), (6400, 256, 256),
        (256, 1024, 257), (900, 512, 300), (4096, 640, 512), (12900, 320, 100), (20000, 256, 200), (22016, 128, 130),
        (4096, 320, 900), (2000, 1600, 40), (2304, 1344, 70), (3900, 11008, 60),
        # more than two accumulations per CTA, added up as they end: of one k-block, of several, of unequal lengths
        (100, 2112, 20), (256, 11008, 130), (768, 3072, 64), (768, 3072, 128), (11264, 2048, 200), (700, 4096, 600),
        # CTA pairs: two shares of k-blocks, an odd number of weight tiles, more tiles than SMs, 128-token tiles
        (4096, 1024, 512), (3968, 1024, 500), (3970, 1024, 256), (20000, 1024, 200), (22016, 512, 256), (12160, 3136, 70),
        (20400, 3200, 120),
        # CTA pairs on a fixed grid: split tiles of many k-blocks, odd numbers of tiles, a partial last one
        (9856, 1088, 700), (20000, 1024, 260), (19500, 704, 300)]


@pytest.mark.parametrize("M,K,T", GEMM)
def test_gemm_paths(ats, M, K, T):
    W, X = _randn((M, K), M + K), _x(T, K, T)
    ref = X[:T].double() @ W.double().T
    # fp32 accumulation of exact bf16 products, the bound of the fp64 comparison of the GEMM
    tol = 4e-5 * K ** 0.5 * float(W.abs().max()) * float(X[:T].abs().max()) + 1e-6
    Y = torch.full((T + 1, M + 3), 7.0, device="cuda")   # a wider output: nothing beyond [T][M] is written
    lib = ats.load()
    from paper_2410_05165_gb300.binding import op_workspace
    st = torch.cuda.current_stream().cuda_stream
    for acc in (0, 1):
        assert lib.atspeed_op_gemm(st, W.data_ptr(), X.data_ptr(), M, K, T, X.shape[0], Y.data_ptr(), M + 3, acc,
                                   op_workspace().data_ptr()) == ats.OK
        want = ref if acc == 0 else 2 * ref
        assert float((Y[:T, :M].double() - want).abs().max()) <= (1 + acc) * tol
        assert bool((Y[T:] == 7).all()) and bool((Y[:, M:] == 7).all())
    assert ats.op_status() == ats.OK


@pytest.mark.parametrize("F,K,T", [(64, 64, 1), (192, 128, 16), (320, 512, 33), (1408, 1024, 128), (1024, 4096, 130),
                                   (3072, 768, 257), (11008, 256, 250), (9728, 192, 40), (5632, 128, 700),
                                   (6080, 128, 120), (9792, 128, 70), (960, 512, 400),
                                   (9920, 192, 200), (5632, 2048, 200), (5632, 2048, 90)])
def test_swiglu_paths(ats, F, K, T):
    W, X = _randn((2 * F, K), F + K, 0.05), _x(T, K, T)
    g, u = (X[:T].double() @ W.double().T).split(F, 1)
    ref = torch.nn.functional.silu(g) * u
    out = ats.op_gemm_swiglu(W, X, T).double()
    # one bf16 unit in the last place, and the fp32 error of g and u carried through the product
    assert bool(((out - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4 * (g.abs() + u.abs() + 1)).all())


# The error of a sum grows with the length of an accumulation in the tensor core (which rounds towards zero), so
# no shape may accumulate longer than a split of its k-blocks over all SMs does: the relative error against fp64
# that this split (one CTA per SM, 152 of them) has on the same inputs, and 3% for another seed.
@pytest.mark.parametrize("M,K,T,limit", [(768, 768, 10, 9.42e-8), (768, 3072, 120, 1.49e-7), (768, 3072, 512, 2.27e-7),
                                         (128, 11008, 200, 2.36e-7), (256, 11008, 10, 2.12e-7), (1024, 11008, 100, 5.44e-7),
                                         (1536, 8192, 40, 6.0e-7), (11264, 2048, 120, 9.77e-7), (22016, 4096, 200, 4.15e-6),
                                         (33024, 4096, 10, 3.72e-6), (33024, 768, 120, 6.17e-7), (22016, 512, 200, 4.44e-7)])
def test_gemm_error_against_fp64(ats, M, K, T, limit):
    W, X = _randn((M, K), M + K, 0.02), _x(T, K, T)
    ref = X[:T].double() @ W.double().T
    assert float((ats.op_gemm(W, X, T).double() - ref).norm() / ref.norm()) <= 1.03 * limit


@pytest.mark.parametrize("M,K", [(2304, 768), (8192, 512), (6400, 256), (20000, 256), (768, 3072), (256, 11008),
                                 (11264, 2048), (8192, 1024), (12288, 4096), (22016, 4096), (22016, 448)])
def test_gemm_result_does_not_depend_on_the_token_count(ats, M, K):
    W, X = _randn((M, K), 5), _x(256, K, 6)
    full = ats.op_gemm(W, X, 256)
    for T in (1, 10, 16, 33, 64, 100, 120, 129, 200):
        assert torch.equal(ats.op_gemm(W, X, T), full[:T])


@pytest.mark.parametrize("F,K", [(320, 512), (5632, 2048), (11008, 512)])
def test_swiglu_result_does_not_depend_on_the_token_count(ats, F, K):
    W, X = _randn((2 * F, K), 5, 0.05), _x(256, K, 6)
    full = ats.op_gemm_swiglu(W, X, 256)
    for T in (1, 33, 64, 128, 200):
        assert torch.equal(ats.op_gemm_swiglu(W, X, T), full[:T])


@pytest.mark.parametrize("T,d", [(1, 4), (7, 256), (9, 260), (3, 1024), (17, 1028), (5, 4096), (2, 4100), (3, 8192),
                                 (2, 8196), (4, 63), (1217, 132)])
@pytest.mark.parametrize("pad", [0, 1])
def test_rmsnorm_paths(ats, T, d, pad):
    h, g = _randn((T, d), T + d, 3.0, torch.float32), _randn((d,), d, 0.1) + 1
    x = torch.full((T, d + pad), 7.0, device="cuda", dtype=torch.bfloat16)
    lib = ats.load()
    assert lib.atspeed_op_rmsnorm(torch.cuda.current_stream().cuda_stream, h.data_ptr(), g.data_ptr(), T, d, 1e-6,
                                  x.data_ptr(), d + pad) == ats.OK
    hd = h.double()
    ref = hd / torch.sqrt(hd.square().mean(1, keepdim=True) + 1e-6) * g.double()
    # half a bf16 unit in the last place of the exact value, and fp32 rounding before it
    assert bool(((x[:, :d].double() - ref).abs() <= (2.0 ** -8 + 1e-6) * ref.abs() + 1e-30).all())
    assert bool((x[:, d:] == 7).all())


# clusters of 4 (few tiles), 2 and 1 (enough tiles and heads), fewer pages than CTAs, no history at all, queries
# that see part of it, with and without path keys (one kernel writes its rows directly), tables of each size
@pytest.mark.parametrize("H,hd,P,T,paths", [(4, 32, 256, 1, True), (2, 64, 1000, 130, True), (3, 128, 64, 17, True),
                                            (5, 64, 128, 63, False), (32, 128, 200, 330, True), (40, 32, 300, 250, True),
                                            (32, 64, 130, 650, True), (32, 128, 321, 641, False), (2, 32, 0, 5, True),
                                            (1, 128, 2100, 64, True), (80, 32, 70, 257, False), (2, 32, 70, 1300, True),
                                            (3, 64, 200, 7700, False), (12, 64, 1000, 1000, False), (4, 32, 1000, 700, False),
                                            # (many CTAs per SM: warps that run late still read their own Q and K/V tiles)
                                            (120, 32, 128, 256, True), (32, 32, 300, 1024, True), (120, 64, 500, 256, True),
                                            (120, 32, 200, 256, False), (32, 32, 1000, 1000, False)])
def test_attention_paths(ats, H, hd, P, T, paths):
    rng = np.random.default_rng(H + P + T)
    d, n = H * hd, (P + 63) // 64
    pages = rng.permutation(n + 3)[:n]
    rows = 64 * (n + 3) + 40
    q, kc = _randn((T, d), T), _randn((rows, d), P)
    vc = _randn((rows, d), P + 1).to(torch.float16)
    vis = np.where(rng.random(T) < 0.5, P, rng.integers(0, P + 1, size=T)).astype(np.int32)
    n_path = rng.integers(0, 5, size=T).astype(np.int32) if paths else None
    path = rng.integers(0, rows, size=(T, 4)).astype(np.int32) if paths else None
    out = ats.op_attention(q, kc, vc, H, hd, P, pages, vis, path, n_path).double().reshape(T, H, hd)
    prefix = torch.from_numpy((64 * pages[:, None] + np.arange(64)).reshape(-1)[:P].astype(np.int64)).cuda()
    heads = lambda t: t.double().reshape(-1, H, hd)   # noqa: E731
    s = torch.einsum("thd,khd->htk", heads(q), heads(kc[prefix]))
    s = s.masked_fill(~(torch.arange(P)[None, :] < torch.from_numpy(vis)[:, None]).cuda(), float("-inf"))
    v = heads(vc[prefix])
    num_v, num_a = [v.transpose(0, 1)], [v.abs().transpose(0, 1)]
    if paths:
        pk, pv = [heads(c[torch.from_numpy(path.astype(np.int64)).cuda().reshape(-1)]).reshape(T, 4, H, hd) for c in (kc, vc)]
        sp = torch.einsum("thd,tjhd->htj", heads(q), pk)
        sp = sp.masked_fill(~(torch.arange(4)[None, :] < torch.from_numpy(n_path)[:, None]).cuda(), float("-inf"))
        s = torch.cat([s, sp], 2)
    w = torch.nan_to_num(torch.softmax(s / hd ** 0.5, 2))   # no key at all: zero
    ref, mag = [torch.einsum("htk,hkd->thd", w[:, :, :P], x[0]) for x in (num_v, num_a)]
    if paths:
        ref = ref + torch.einsum("htj,tjhd->thd", w[:, :, P:], pv)
        mag = mag + torch.einsum("htj,tjhd->thd", w[:, :, P:], pv.abs())
    # the weights are rounded to fp16 (2^-11), the result to bf16
    assert bool(((out - ref).abs() <= 2.0 ** -8 * ref.abs() + 2.0 ** -11 * mag + 1e-5).all())


# tables on both sides of what kernel parameters hold: nothing beyond the scratch that the call asks for is written
@pytest.mark.parametrize("T", [1200, 1300])
def test_attention_scratch(ats, T):
    H, hd, P = 2, 32, 70
    d, rows, rng = H * hd, 64 * 4, np.random.default_rng(T)
    q, kc = _randn((T, d), 1), _randn((rows, d), 2)
    vc = _randn((rows, d), 3).to(torch.float16)
    pages, vis = np.array([2, 0], np.int32), rng.integers(0, P + 1, size=T).astype(np.int32)
    n_path, path = rng.integers(0, 5, size=T).astype(np.int32), rng.integers(0, rows, size=(T, 4)).astype(np.int32)
    lib = ats.load()
    size = lib.atspeed_op_attention_scratch(T, H, hd, P)
    part, out = torch.full((size + 256,), 7, dtype=torch.uint8, device="cuda"), torch.empty_like(q)
    ptr = [x.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)) for x in (pages, vis, path, n_path)]
    assert lib.atspeed_op_attention(torch.cuda.current_stream().cuda_stream, q.data_ptr(), kc.data_ptr(), vc.data_ptr(),
                                    rows, T, H, hd, P, *ptr, out.data_ptr(), part.data_ptr()) == ats.OK
    assert bool((part[size:] == 7).all())
    assert torch.equal(out, ats.op_attention(q, kc, vc, H, hd, P, pages, vis, path, n_path))
    assert ats.op_status(noalloc=True) == ats.OK   # (no bounded wait gave up: the attention's word is among these)


# up to 256 tokens a query's result is that of its own keys, whatever else is in the call: fewer queries, other
# tiles, neighbours that see more or less of the prefix; the numbers of heads and pages that give one, two and
# four splits
@pytest.mark.parametrize("H,hd,P", [(32, 128, 448), (32, 128, 512), (32, 64, 200), (4, 32, 250), (12, 64, 1000), (60, 32, 600),
                                    (120, 32, 300), (2, 64, 2500)])
def test_attention_result_does_not_depend_on_the_other_queries(ats, H, hd, P):
    rng = np.random.default_rng(P)
    T, d, n = 256, H * hd, (P + 63) // 64
    pages = rng.permutation(n + 3)[:n]
    rows = 64 * (n + 3) + 40
    q, kc = _randn((T, d), 1), _randn((rows, d), 2)
    vc = _randn((rows, d), 3).to(torch.float16)
    vis = np.where(rng.random(T) < 0.5, P, rng.integers(0, P + 1, size=T)).astype(np.int32)
    n_path = rng.integers(0, 5, size=T).astype(np.int32)
    path = rng.integers(0, rows, size=(T, 4)).astype(np.int32)
    n_path[[7, 60]] = 4   # (path keys in every call of the first kind)

    def run(i, paths):
        i = np.asarray(i)
        return ats.op_attention(q[torch.from_numpy(i).cuda()].contiguous(), kc, vc, H, hd, P, pages, vis[i],
                                path[i] if paths else None, n_path[i] if paths else None)

    for paths in (True, False):
        full = run(np.arange(T), paths)
        for i in ([7], np.arange(10), np.concatenate([[7], rng.permutation(T)[:63]]), np.arange(120), np.arange(50, 250)):
            assert torch.equal(run(i, paths), full[torch.as_tensor(i).cuda()])


# whole-vocabulary log-sum-exp (FULL normalisation): one token tile of every width, several; a partial last
# weight tile; enough tiles for the CTA pairs on a fixed grid (an odd and an even count), pairs of 128- and
# 256-token tiles, more than two accumulations
@pytest.mark.parametrize("V,users,N,gamma,d", [(1200, 1, 7, 1, 64), (1200, 3, 17, 1, 64), (2000, 2, 40, 1, 64),
                                               (1200, 1, 80, 3, 64), (1025, 3, 100, 3, 64), (33024, 1, 100, 3, 64),
                                               (16500, 4, 100, 3, 64), (9700, 2, 100, 1, 512), (16384, 1, 100, 1, 3072),
                                               (33024, 1, 80, 3, 512), (1300, 1, 40, 1, 3072)])
def test_full_lse_paths(ats, V, users, N, gamma, d):
    from types import SimpleNamespace
    f = 128
    w = {"embed": _randn((V, d), 1), "lm_head": _randn((V, d), 2, 3.2 / d ** 0.5), "final_norm": _randn((d,), 3, 0.1) + 1}
    for name, shape in (("attn_norm", (d,)), ("mlp_norm", (d,)), ("wqkv", (3 * d, d)), ("wo", (d, d)),
                        ("wgate_up", (2 * f, d)), ("wdown", (d, f))):
        w["layers.0." + name] = _randn(shape, 4 + len(name), 0.1)
    spec = SimpleNamespace(n_layers=1, d_model=d, n_heads=max(2, d // 128), d_ffn=f, vocab=V, rms_eps=1e-6, rope_theta=1e4)
    items = np.zeros((256, 4), np.int32)
    items[:, 0] = np.arange(256)
    ctx = ats.Context(spec, w, None, None, items, 0, max_users=users, max_prompt=8, max_K=5, max_N=N, max_gamma=gamma)
    o = ats.opts(5, N, gamma, norm=ats.NORM_FULL)
    ctx.prefill(torch.arange(8 * users, dtype=torch.int32, device="cuda"), 8 * np.arange(users + 1))
    ctx.begin_step(o)
    parents, codes = np.zeros((2, users, gamma, N), np.int32)
    parents[:, 1:], codes[:, 0] = np.arange(N), np.arange(N)
    ctx.set_tree(np.full((users, gamma), N), parents, codes, np.zeros((users, gamma, N)))
    ctx.verify(o, ats.STRICT)
    T = users * gamma * N
    x = torch.from_numpy(ctx.debug_buffer(0, 1, np.int16, T * d).reshape(T, d)).cuda().view(torch.bfloat16)
    ref = torch.logsumexp(x.double() @ w["lm_head"].double().T, 1)
    got = torch.from_numpy(ctx.debug_buffer(0, 10, np.float32, users + T)[users:]).cuda().double()
    # fp32 logits (|x . w| up to ~30) and exponentials of them: a few units of 2^-23 of the largest logit; each of the
    # d / 16 steps of a long accumulation truncates it once
    assert float((got - ref).abs().max()) < max(2e-5, d / 16 * 2.0 ** -23 * 30)
    ctx.close()


# forwards of more than 256 tokens: split tiles are split for as many CTAs as a 256-token forward has, however
# many run; 2048 and 4096 tokens of this model (6 to 48 weight tiles, split for 48 CTAs) are whole tiles alone, so
# a user's logits do not depend on the other users'
def test_long_forward_sums_do_not_depend_on_the_grid(ats):
    from types import SimpleNamespace
    d, f, V, P = 768, 3072, 1024, 1024
    w = {"embed": _randn((V, d), 1), "lm_head": _randn((V, d), 2, 0.1), "final_norm": _randn((d,), 3, 0.1) + 1}
    for name, shape in (("attn_norm", (d,)), ("mlp_norm", (d,)), ("wqkv", (3 * d, d)), ("wo", (d, d)),
                        ("wgate_up", (2 * f, d)), ("wdown", (d, f))):
        w["layers.0." + name] = _randn(shape, 4 + len(name), 0.02) + (1 if "norm" in name else 0)
    spec = SimpleNamespace(n_layers=1, d_model=d, n_heads=12, d_ffn=f, vocab=V, rms_eps=1e-6, rope_theta=1e4)
    items = np.zeros((256, 4), np.int32)
    items[:, 0] = np.arange(256)
    tokens = torch.from_numpy(np.random.default_rng(0).integers(0, V, 4 * P).astype(np.int32)).cuda()
    ctx = ats.Context(spec, w, None, None, items, 0, max_users=4, max_prompt=P, max_K=5, max_N=10, max_gamma=1)
    got = []
    for users in (2, 4):
        ctx.prefill(tokens[:users * P], P * np.arange(users + 1))
        got.append(ctx.debug_buffer(0, 7, np.float32, 2 * 1024).copy())
    assert np.array_equal(*got)
    ctx.close()


# the exact selection of a drafted level (score descending, index ascending): one histogram pass, several (an
# outlier widens the range), none (few candidates), more equal keys than are ranked at once, infinite scores
@pytest.mark.parametrize("N", [1, 5, 40, 100])
@pytest.mark.parametrize("kind", ["spread", "outlier", "equal", "three", "inf", "few"])
def test_selection_paths(ats, kind, N):
    from types import SimpleNamespace
    d, f, V = 64, 128, 1024
    w = {"embed": _randn((V, d), 1), "lm_head": _randn((V, d), 2, 0.4), "final_norm": _randn((d,), 3, 0.1) + 1}
    for name, shape in (("attn_norm", (d,)), ("mlp_norm", (d,)), ("wqkv", (3 * d, d)), ("wo", (d, d)),
                        ("wgate_up", (2 * f, d)), ("wdown", (d, f))):
        w["layers.0." + name] = _randn(shape, 4 + len(name), 0.1)
    spec = SimpleNamespace(n_layers=1, d_model=d, n_heads=2, d_ffn=f, vocab=V, rms_eps=1e-6, rope_theta=1e4)
    n = 7 if kind == "few" else 256
    items = np.zeros((n * n, 4), np.int32)
    items[:, 0], items[:, 1] = np.repeat(np.arange(n), n), np.tile(np.arange(n), n)
    rng = np.random.default_rng(N)
    # logits of the two levels, the same for every parent: different sums differ by 2^-8 at least, beyond fp32
    # rounding, so the order of the sums is that of the scores
    x = [rng.permutation(256) * 1.0, rng.permutation(256) / 256.0]
    if kind == "outlier":
        x = [1 + rng.permutation(256) / 256.0, rng.permutation(256) * 1.0]
        x[0][3] = x[1][200] = -10000.0
    elif kind == "equal":
        x = [np.full(256, 1.25)] * 2
    elif kind == "three":
        x = [np.array([0.0, 1.0, 3.0])[rng.integers(0, 3, 256)] for _ in range(2)]
    elif kind == "inf":
        for v in x:
            v[rng.permutation(256)[:250]] = -np.inf
    ctx = ats.Context(spec, w, spec, w, items, 0, max_users=1, max_prompt=8, max_K=1, max_N=N, max_gamma=2)
    o = ats.opts(1, N, 2)
    ctx.prefill(torch.arange(8, dtype=torch.int32, device="cuda"), [0, 8])
    ctx.begin_step(o)
    beams, score = [()], np.zeros(1)
    for lvl in range(2):
        tree = ctx.debug_tree(2)
        width = tree["slots_in"] if lvl == 0 else tree["slots_lvl"]
        ctx.draft_step_logits(o, ats.STRICT, np.tile(np.tile(x[lvl], 4).astype(np.float32), (1, width, 1)))
        s = (score[:, None] + x[lvl][None, :n]).reshape(-1)
        order = np.lexsort((np.arange(s.size), -s))[:N]
        beams, score = [beams[i // n] + (i % n,) for i in order], s[order]
        tree = ctx.debug_tree(2)
        off = tree["slots_in"] + lvl * tree["slots_lvl"]
        assert tree["count"][0, lvl + 1] == len(order)
        got = [tuple(int(c) for c in q if c >= 0) for q in tree["path"][0, off:off + len(order)]]
        assert got == beams
    ctx.close()
