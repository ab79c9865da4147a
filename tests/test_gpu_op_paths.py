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
