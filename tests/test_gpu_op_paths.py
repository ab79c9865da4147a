"""Each path of the operators' dispatch at the sizes where it can go wrong (edges of tiles, groups and
cluster sizes, the smallest and largest of a range, general alignments) against fp64."""
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
        (4096, 320, 900)]


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
                                   (3072, 768, 257), (11008, 256, 250), (9728, 192, 40), (5632, 128, 700)])
def test_swiglu_paths(ats, F, K, T):
    W, X = _randn((2 * F, K), F + K, 0.05), _x(T, K, T)
    g, u = (X[:T].double() @ W.double().T).split(F, 1)
    ref = torch.nn.functional.silu(g) * u
    out = ats.op_gemm_swiglu(W, X, T).double()
    # one bf16 unit in the last place, and the fp32 error of g and u carried through the product
    assert bool(((out - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4 * (g.abs() + u.abs() + 1)).all())


def test_gemm_result_does_not_depend_on_the_token_count(ats):
    M, K = 2304, 768
    W, X = _randn((M, K), 5), _x(256, K, 6)
    full = ats.op_gemm(W, X, 256)
    for T in (1, 16, 33, 100, 129, 200):
        assert torch.equal(ats.op_gemm(W, X, T), full[:T])


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
