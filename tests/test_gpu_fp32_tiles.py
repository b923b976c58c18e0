"""The fp32 row GEMMs with one, two, four and eight warps to a warp tile and one and two groups to a block tile, and the search
for a row tile among more experts than a warp has lanes.  (Four warps: the other fp32 tests.)"""
import pytest
import torch

from test_gpu_kernel_edges import test_fp32_expert_ffn_at_the_edges_of_its_tiles as check_ffn
from test_gpu_kernel_edges import test_fp32_router_products_at_the_edges_of_their_tiles as check_router

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,d,f", [
    ([7, 0, 33, 1, 8, 0, 2, 13] * 5, 128, 768),             # gate/up: two warps to a tile; 40 experts
    ([64, 0, 1, 31, 32, 33, 95, 96, 97, 0, 128] * 3, 256, 1024),       # one; groups that end on tiles of 32
    ([0, 20], 320, 640),                                    # eight, which 20 chunks do not divide among evenly
    ([1] * 65 + [0] * 30 + [2], 192, 256),                  # 96 experts: three rounds of the search
    # warp tiles, groups of fewer than 96 rows
    ([64, 31, 95, 33, 1, 96, 100, 60] * 5, 128, 768),       # one warp: gate/up (misaligned: block tiles)
    ([64, 31, 95, 33, 1, 96, 100, 60] * 5, 1024, 256),      # one warp: down
    ([64, 31, 95, 33, 1, 96, 100, 60] * 5, 768, 512),       # two warps, a contraction of 768: gate/up
    ([64, 31, 95, 33, 1, 96, 100, 60] * 5, 1024, 768),      # two warps, a contraction of 768: down, gate/up
    ([25, 0, 50, 24] * 10, 1024, 64),                       # two warps, a short contraction: down
    # block tiles; groups that end at and beside tiles of 64
    ([200, 0, 64, 511, 321, 129, 128, 1, 65, 63, 448, 470], 128, 768),   # one group: gate/up
    ([362, 0, 896, 65, 300, 400, 449, 460], 1024, 64),      # one group: down, dgrad gate/up
    ([362, 0, 896, 65, 300, 400, 449, 460], 1024, 256),     # two groups: down, dgrad gate/up
    ([127, 513, 0, 321], 768, 1536),                        # two groups, a contraction of 768: gate/up
    ([1000, 577, 1, 1022, 640, 770], 128, 1536),            # one group: dgrad down
    ([1000, 577, 1, 1022, 640, 770], 768, 1536),            # two groups: dgrad down
    ([1311] * 400, 64, 64),                                 # more than 8192 row tiles
])
@pytest.mark.parametrize("shift", [0, 1])
def test_fp32_ffn_by_tiles(sizes, d, f, shift):
    check_ffn(sizes, d, f, shift)


def test_fp32_rows_of_padded_groups_are_the_same():
    """Without the group sizes all tiles of the padded groups are multiplied: zeros stay zeros, the rest is the same sums."""
    from paper_2605_06665_b200 import binding as B
    M, d, f, T = 37, 128, 192, 900
    ctx = B.Context(B.make_config(d, f, M, 1, 1, T, B.FP32, 1e-6, 2.0))
    cap, g = ctx.row_capacity, torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(T, d, device="cuda", generator=g)
    Wgu, Wd = (torch.randn(*s, device="cuda", generator=g) * 0.05 for s in ((M, 2 * f, d), (M, d, f)))
    idx = torch.randint(0, M, (T, 1), device="cuda", generator=g).to(torch.int32)
    off, row_of, tok, te, rows = (torch.empty(s, dtype=torch.int32, device="cuda")
                                  for s in ((M + 1,), (T, 1), (cap,), (cap // 128,), (M,)))
    Xp = torch.empty(cap, d, device="cuda")
    ctx.dispatch(x, T, idx, M, off, row_of, tok, te, Xp, rows)
    out = []
    for r in (rows, None):
        out.append([torch.full((cap, w), float("nan"), device="cuda") for w in (2 * f, f, d)])
        ctx.expert_fwd(Xp, off, te, Wgu, Wd, 0, M, *out[-1], r)
    used = int(off[-1])
    for a, b in zip(*out):
        assert torch.equal(a[:used], b[:used]) and a[used:].isnan().all() and b[used:].isnan().all()
    ctx.check_status()
    ctx.close()


@pytest.mark.parametrize("T,M,d", [
    (148 * 32, 16, 64), (148 * 32 + 1, 64, 64),             # 148 and 149 tiles of logits: eight and four warps to each
    (3 * 8 * 148, 65, 128), (3 * 8 * 148 + 1, 65, 128), (8 * 8 * 148, 10, 64), (8 * 8 * 148 + 1, 10, 64),   # one, four tokens to a selecting warp
    (2000, 300, 192), (37, 512, 128),
])
@pytest.mark.parametrize("shift", [0, 1])
def test_fp32_router_by_tiles(T, M, d, shift):
    check_router(T, M, d, shift)
